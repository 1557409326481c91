"""The diagonal-resolved trispectrum where its pair spectra take several groups
(FBS_DIAG_GROUP: pairs of a group) and where device memory is short: the same
results as with one group and all the scratch it asks for."""
import math

import numpy as np
import pytest
import torch

import fields
import paper_1705_06284_gb300 as fbs
from test_diagonal_gpu import _diag_edges, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [1, 2, 3, 7])
def test_groups_of_pairs(pairs, monkeypatch):
    N, L = 32, 100.0
    edges = fields.linear_edges(N, L, 5)
    dedges = _diag_edges(N, L, 6)
    f32 = fields.quadratic_local(N, 1.0, -1.5, 0.3, seed=84).astype(np.float32)
    with fbs.Plan(N, L, edges, precision="fp32", trispectrum=True) as plan:
        assert len({tuple(q[:2]) for q in plan.quads} | {tuple(q[2:]) for q in plan.quads}) > 7
        plan.set_diagonal(dedges)
        one = plan.trispectrum_diagonal(f32)
        monkeypatch.setenv("FBS_DIAG_GROUP", str(pairs))
        assert np.array_equal(plan.trispectrum_diagonal(f32), one, equal_nan=True)
        g, r, _, _ = _run(plan, f32, L, edges, dedges)
    assert g.sum() >= 10 and r[g].max() < 1e-4


@pytest.mark.parametrize("N,nb,nd", [(48, 12, 12), (64, 14, 4)])
def test_short_of_memory(N, nb, nd):
    """Within what the fields, one product, its transforms and the pair spectra take."""
    L = 2.0 * N
    edges = fields.linear_edges(N, L, nb)
    dedges = _diag_edges(N, L, nd)
    f = torch.from_numpy(fields.quadratic_local(N, 1.0, -1.5, 0.3, seed=85).astype(np.float32)).cuda()
    with fbs.Plan(N, L, edges, precision="fp32", trispectrum=True, single_grid=True) as plan:
        plan.set_diagonal(dedges)
        TD = torch.zeros(plan.nquad * nd, dtype=torch.float64, device="cuda")
        full = plan.trispectrum_diagonal(f, TD).cpu().numpy().copy()
        M = plan.levels[0]["M"]
        R = [min(math.isqrt(int(t) - 1), M // 2) for t in plan.thresholds[1:]]
        Rq = min(math.isqrt(round((dedges[-1] * L / (2 * math.pi)) ** 2) - 1), M // 2)
        D, Dz = min(2 * Rq + 1, M), Rq + 1
        np_ = len({tuple(q[:2]) for q in plan.quads} | {tuple(q[2:]) for q in plan.quads})
        need = 4 * nb * M ** 3 + 8 * sum(M * M * (r + 1) for r in R) + 4 * nb * M * M  # fields, y stage, squares
        need += 4 * M ** 3 + 8 * (M * M * Dz + M * D * Dz) + 8 * np_ * D * D * Dz + 64
        fbs.fbs_set_device_budget(fbs.fbs_device_bytes_in_use() + need)
        try:
            tight = plan.trispectrum_diagonal(f, TD).cpu().numpy()
        finally:
            fbs.fbs_set_device_budget(0)
    assert np.array_equal(tight, full, equal_nan=True)
