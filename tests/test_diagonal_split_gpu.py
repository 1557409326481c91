"""The diagonal-resolved trispectrum where its work split changes: more
quadruplets than one thread each holds, pair products read by both forward z
passes (compile-time and run-time grids), a single diagonal shell and many;
against the oracle as in test_diagonal_gpu."""
import numpy as np
import pytest

import fields
import paper_1705_06284_gb300 as fbs
from test_diagonal_gpu import _diag_edges, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nb,nd", [(32, 8, 9), (48, 9, 3), (64, 7, 2)])
def test_many_quadruplets(N, nb, nd):
    L = 2.0 * N
    edges = fields.linear_edges(N, L, nb)
    f32 = fields.quadratic_local(N, 1.0, -1.5, 0.3, seed=83).astype(np.float32)
    with fbs.Plan(N, L, edges, precision="fp32", trispectrum=True) as plan:
        g, r, _, _ = _run(plan, f32, L, edges, _diag_edges(N, L, nd))
        assert plan.nquad > 128
    assert g.sum() >= 10 and r[g].max() < 1e-4
