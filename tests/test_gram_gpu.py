"""The shared-operand tensor-core contraction (the default of BF16x3 plans)
where its layouts change: one and two accumulator tiles, rows of operand A
alone, several CTA groups, partial last steps, batches; against the FP64
oracle within the BF16x3 gate (2e-4)."""
import numpy as np
import pytest

import fields
import oracle
import paper_1705_06284_gb300 as fbs
from gpu_util import check_bispectrum, check_trispectrum

pytestmark = pytest.mark.gpu


def _shape(plan):
    return [j for lvl in plan.tc_info() for j in lvl.values()]


@pytest.mark.parametrize("N,nb,kind,tiles", [(24, 3, "lin", 1), (64, 16, "log", 1), (72, 16, "lin", 2), (54, 9, "log", 1)])
@pytest.mark.parametrize("planes", [0, 1])
def test_triplets_and_quadruplets(N, nb, kind, tiles, planes):
    """planes = 1: slabs of one plane, whose points are no multiple of a step
    (54^2) or fewer than one flush."""
    import torch
    L = 1.5 * N
    edges = fields.linear_edges(N, L, nb) if kind == "lin" else fields.log_edges(N, L, nb)
    f32 = fields.quadratic_local(N, 0.5, -1.5, 0.3, seed=91).astype(np.float32)
    with fbs.Plan(N, L, edges, precision="bf16x3", trispectrum=True, single_grid=True) as plan:
        plan.set_option(fbs.FBS_OPT_SLAB_PLANES, planes)
        T, B, P = plan.trispectrum(torch.from_numpy(f32).cuda())
        plan.check()
        info = _shape(plan)
        assert [j["tiles"] for j in info] == [tiles] and info[0]["stages"][0] == 0
        check_trispectrum(plan, T.cpu().numpy(), f32, L, edges, 2e-4)
        if nb <= 9:
            check_bispectrum(plan, B.cpu().numpy(), P.cpu().numpy(), f32, L, edges, "bf16x3")


@pytest.mark.parametrize("N,nb", [(32, 5), (64, 15), (72, 33), (96, 48)])
def test_triplets(N, nb):
    """Pairs as operand A (few bins), single bins as operand A (one and several CTA groups)."""
    import torch
    L = 2.0 * N
    edges = fields.linear_edges(N, L, nb)
    f32 = fields.lognormal(N, 0.6, -1.5, seed=92).astype(np.float32)
    f = torch.from_numpy(f32).cuda()
    with fbs.Plan(N, L, edges, precision="bf16x3") as plan:
        B, P = plan.bispectrum(f)
        plan.check()
        assert all(j["stages"][0] == 0 for j in _shape(plan))
        ref = oracle.fft_estimator(f32.astype(np.float64), L, edges, triplets=plan.triplets)
        g = (plan.N_tri >= 100) & (np.abs(ref["B"]) >= 1e-3 * ref["M"])
        assert np.max(np.abs(B.cpu().numpy() - ref["B"])[g] / np.abs(ref["B"])[g]) < 2e-4
        Bb, _ = plan.bispectrum_batch([f, f, f])
        assert np.max(np.abs(Bb.cpu().numpy() - ref["B"])[:, g] / np.abs(ref["B"])[g]) < 2e-4
        assert torch.equal(Bb[0], Bb[2])
