"""fbs_plan_tc_info reports the launches there were and changes nothing: no
tables built, no device memory taken, whatever the device budget leaves."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import numpy as np, torch
import fields
import paper_1705_06284_gb300 as fbs
N, L = 32, 32.0
f = torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=3).astype(np.float32)).cuda()
for tri in (False, True):
    with fbs.Plan(N, L, fields.linear_edges(N, L, 5), precision="bf16x3", trispectrum=tri) as plan:
        B, P = plan.bispectrum(f)
        torch.cuda.synchronize()
        used = fbs.fbs_device_bytes_in_use()
        fbs.fbs_set_device_budget(used)
        info = plan.tc_info()
        fbs.fbs_set_device_budget(0)
        assert fbs.fbs_device_bytes_in_use() == used
        assert set(info[0]) == {"triplets"}, info
print("unchanged")
"""


def test_query_takes_no_memory():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=root))
    assert r.returncode == 0 and "unchanged" in r.stdout, r.stderr[-2000:]
