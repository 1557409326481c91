"""The general plan where its work split changes: odd and uneven sides, more
items than a block's threads, empty bins, one bin; against the FP64 oracle
within 1e-4 as in test_general_gpu, and sums past FP32's range."""
import math

import numpy as np
import pytest

import oracle
import paper_1705_06284_gb300 as fbs
from test_general_gpu import _edges, _field, _scale

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,nb", [((27, 16, 81), 3), ((16, 27, 27), 4), ((16, 54, 24), 14), ((32, 8, 36), 1), ((18, 96, 12), 5)])
def test_matches_oracle(shape, nb):
    Ls = tuple(1.7 * n * s for n, s in zip(shape, (1.0, 1.1, 0.9)))
    f = _field(shape, "complex", 51)
    edges = _edges(shape, Ls, nb)
    with fbs.GeneralPlan(shape, Ls, edges) as plan:
        ref = oracle.general_bispectrum(f.astype(np.complex128), Ls, edges)
        assert np.array_equal(plan.triplets, ref["triplets"]) and np.array_equal(plan.shell, ref["shell"])
        B, P = plan.bispectrum(f)
        # the same field twice as large: exactly 8 and 4 times the estimates
        B2, P2 = plan.bispectrum(f * np.float32(2))
        ok = ref["shell"] > 0
        assert np.array_equal(B2, 8 * B) and np.array_equal(P2[ok], 4 * P[ok])
    assert np.all(np.abs(P[ok] - ref["P"][ok]) <= 1e-4 * np.abs(ref["P"][ok]))
    if len(ref["B"]):
        M = _scale(f, Ls, edges, ref["triplets"]) / np.maximum(ref["N_tri"], 1)
        g = (ref["N_tri"] >= 100) & (np.abs(ref["B"]) >= 1e-3 * M)
        assert np.all(np.abs(B - ref["B"])[g] <= 1e-4 * np.abs(ref["B"])[g])


def test_sums_past_the_range_of_fp32():
    """Products near 1e37 whose sums pass 3.4e38: FP64 totals, not infinities."""
    shape, Ls = (32, 32, 32), (10.0, 10.0, 10.0)
    f = _field(shape, "real", 52)
    edges = _edges(shape, Ls, 3)
    with fbs.GeneralPlan(shape, Ls, edges) as plan:
        B, P = plan.bispectrum(f)
        D = np.fft.fftn(f.astype(np.float64))
        bins = oracle.general_bin_index(shape, Ls, edges)
        top = max(np.abs(np.fft.ifftn(np.where(bins == b, D, 0)) * f.size).max() for b in range(3))
        s = np.float32(2.0 ** math.floor(math.log2((1e38) ** (1.0 / 3.0) / top)))
        Bs, Ps = plan.bispectrum((f * s).astype(np.float32))
    assert np.all(np.isfinite(Bs)) and np.all(np.abs(Bs / float(s) ** 3 - B) <= 1e-12 * np.abs(B))
