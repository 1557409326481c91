"""Top edges far above the grid's largest |m|: with aliased closure allowed no
edge is refused, and a shell holds what the grid has of it whatever the square
of its edge (past 2^31 from 46,341 k_f on)."""
import numpy as np
import pytest
import torch

import fields
import paper_1705_06284_gb300 as fbs

pytestmark = pytest.mark.gpu


def _available_gb():
    with open("/proc/meminfo") as f:
        return next(int(x.split()[1]) for x in f if x.startswith("MemAvailable")) / 2 ** 20


def test_top_edge_past_32_bits():
    if _available_gb() < 24:
        pytest.skip("plan creation tabulates every |m|^2 below the top edge: 8 GB of host memory")
    N = 64
    L = float(N)
    kf = 2 * np.pi / L
    f = torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=71).astype(np.float32)).cuda()
    got = []
    for top in (60.0, 46342.0):  # both above sqrt(3) N / 2: the same modes
        with fbs.Plan(N, L, np.array([1.0, 3.0, 30.0, top]) * kf, precision="fp32", allow_aliased=True) as plan:
            B, P = plan.bispectrum(f)
            torch.cuda.synchronize()
            got.append((plan.shell.copy(), plan.N_tri.copy(), B.cpu().numpy(), P.cpu().numpy()))
    assert got[0][0][2] > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
