"""Estimates formed by the reduction (plans of one level) and by the separate
normalisation (several levels): empty bins, batches, all three outputs."""
import numpy as np
import pytest
import torch

import fields
import oracle
import paper_1705_06284_gb300 as fbs
from gpu_util import TOL, gate_mask, rel_err, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("single", [True, False])
@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_empty_bins_and_batches(precision, single, monkeypatch):
    N = 96 if single else 144
    L = float(N)
    if not single:
        monkeypatch.setenv("FBS_LEVEL_COST", "-1e15")  # every level its own grid
    edges = np.insert(fields.linear_edges(N, L, 6), 3, fields.linear_edges(N, L, 6)[3])  # bin 3 is empty
    f = [fields.lognormal(N, 0.5, -1.5, seed=700 + i).astype(np.float32) for i in range(2)]
    with fbs.Plan(N, L, edges, precision=precision, single_grid=single) as plan:
        assert (len(plan.levels) == 1) == single and plan.shell[3] == 0
        B, P = run(plan, f[0])
        e = oracle.fft_estimator(f[0].astype(np.float64), L, edges, triplets=plan.triplets)
        ok = plan.shell > 0
        assert np.array_equal(np.isnan(P), ~ok)
        assert np.all(rel_err(P[ok], e["P"][ok]) < 1e-5)
        g = gate_mask(e["B"], e["M"], e["N_tri"])
        assert g.sum() >= 3 and rel_err(B, e["B"])[g].max() < TOL[precision]
        Bb, Pb = plan.bispectrum_batch([torch.from_numpy(v).cuda() for v in f])
        Bb, Pb = [np.asarray(v.cpu() if torch.is_tensor(v) else v) for v in (Bb, Pb)]
        for i in range(2):
            Bi, Pi = run(plan, f[i])
            assert np.array_equal(Pb[i], Pi, equal_nan=True)
            assert np.all(rel_err(Bb[i], Bi)[g] <= 2 * TOL[precision])
