"""The FP32 contraction where its work split changes: fewer pairs than a group
holds, groups split by rows, chunks of 128 to 512 points, ragged tails (slabs
of one plane), many bins and several blocks of items; against the FP64
oracle's FFT estimator within the FP32 gate (1e-4)."""
import numpy as np
import pytest

import fields
import oracle
import paper_1705_06284_gb300 as fbs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nb,quads", [(16, 1, False), (24, 3, True), (54, 9, True), (64, 16, False), (72, 12, True),
                                        (96, 64, False)])
@pytest.mark.parametrize("planes", [0, 1])
def test_sums_match_the_oracle(N, nb, quads, planes):
    import torch
    L = 1.5 * N
    edges = fields.linear_edges(N, L, nb)
    f32 = fields.quadratic_local(N, 0.5, -1.5, 0.3, seed=95).astype(np.float32)
    f = torch.from_numpy(f32).cuda()
    with fbs.Plan(N, L, edges, precision="fp32", trispectrum=quads) as plan:
        plan.set_option(fbs.FBS_OPT_SLAB_PLANES, planes)
        out = plan.trispectrum(f) if quads else plan.bispectrum(f)
        torch.cuda.synchronize()
        B = out[-2].cpu().numpy()
        ref = oracle.fft_estimator(f32.astype(np.float64), L, edges, triplets=plan.triplets)
        g = (plan.N_tri >= 100) & (np.abs(ref["B"]) >= 1e-3 * ref["M"])
        assert g.any() and np.max(np.abs(B - ref["B"])[g] / np.abs(ref["B"])[g]) < 1e-4
        if quads:
            from gpu_util import check_trispectrum
            check_trispectrum(plan, out[0].cpu().numpy(), f32, L, edges, 1e-4)


def test_precision_change_builds_the_tables():
    import torch
    N, L, nb = 32, 40.0, 6
    edges = fields.linear_edges(N, L, nb)
    f = torch.from_numpy(fields.lognormal(N, 0.5, -2.0, seed=4).astype(np.float32)).cuda()
    with fbs.Plan(N, L, edges, precision="bf16x3") as a, fbs.Plan(N, L, edges, precision="fp32") as b:
        a.set_precision("fp32")
        assert torch.equal(a.bispectrum(f)[0], b.bispectrum(f)[0])
