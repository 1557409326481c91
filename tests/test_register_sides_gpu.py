"""The register forward z and inverse x, y and z passes at the remaining grids
they are compiled for: P and B of a full-grid plan against FP64 transforms
(tolerances as for the other grids: 1e-5 on P, 1e-4 on B gated on the
cancellation-free scale)."""
import numpy as np
import pytest
import torch

import fields
import oracle
import paper_1705_06284_gb300 as fbs
from gpu_util import TOL, gate_mask, rel_err, run

pytestmark = pytest.mark.gpu


def _fp64(field, L, edges, triplets):
    """(shell counts, P, triplet counts, B, scale) from cuFFT in FP64."""
    N = field.shape[0]
    V, npix = L ** 3, float(N) ** 3
    D = torch.fft.fftn(torch.from_numpy(field).cuda().double())
    bins = torch.from_numpy(oracle.bin_index(N, oracle.thresholds(edges, L))).cuda()
    shells, counts, nsh, P = [], [], [], []
    for b in range(len(edges) - 1):
        on = bins == b
        Db = torch.where(on, D, 0)
        nsh.append(int(on.sum()))
        P.append(V / npix ** 2 * float((Db.abs() ** 2).sum()) / max(1, nsh[-1]))
        shells.append(torch.fft.ifftn(Db).real * npix)
        counts.append(torch.fft.ifftn(on.double()).real * npix)
    nt = np.array([float((counts[a] * counts[b] * counts[c]).sum()) / npix for a, b, c in triplets])
    c0 = V ** 2 / npix ** 3 / npix
    B = np.array([float((shells[a] * shells[b] * shells[c]).sum()) for a, b, c in triplets]) * c0 / nt
    M = np.array([float((shells[a] * shells[b] * shells[c]).abs().sum()) for a, b, c in triplets]) * c0 / nt
    return np.array(nsh), np.array(P), nt, B, M


@pytest.mark.parametrize("N", [162, 324, 432])
def test_matches_fp64(N):
    L = float(N)
    edges = fields.linear_edges(N, L, 4)
    f32 = fields.lognormal(N, 0.5, -1.5, seed=900 + N).astype(np.float32)
    with fbs.Plan(N, L, edges, precision="fp32", full_grid=True) as plan:
        assert plan.eval_grid == N
        B, P = run(plan, f32)
        nsh, Pr, nt, Br, M = _fp64(f32, L, edges, plan.triplets)
        assert np.array_equal(plan.N_tri, np.rint(nt).astype(np.int64))
        ok = nsh > 0
        assert np.all(rel_err(P[ok], Pr[ok]) < 1e-5)
        g = gate_mask(Br, M, plan.N_tri)
        assert g.sum() >= 1
        assert rel_err(B, Br)[g].max() < TOL["fp32"]
