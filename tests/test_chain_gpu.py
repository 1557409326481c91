"""Evaluations queued back to back (stages launched ahead of their turn below
a size, the ordinary way above it), also from a captured graph: the same
outputs as one evaluation at a time."""
import numpy as np
import pytest
import torch

import fields
import paper_1705_06284_gb300 as fbs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nb,precision", [(32, 6, "fp32"), (64, 12, "bf16x3"), (96, 8, "fp32"), (128, 12, "bf16x3")])
def test_back_to_back(N, nb, precision):
    L = float(N)
    stream = torch.cuda.Stream()
    f = [torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=800 + i).astype(np.float32)).cuda() for i in range(4)]
    torch.cuda.synchronize()
    with fbs.Plan(N, L, fields.linear_edges(N, L, nb), precision=precision, single_grid=True,
                  stream=stream.cuda_stream) as plan, torch.cuda.stream(stream):
        def outputs():
            return (torch.zeros(plan.ntrip, dtype=torch.float64, device="cuda"),
                    torch.zeros(plan.nbins, dtype=torch.float64, device="cuda"))
        one = []
        for x in f:
            B, P = outputs()
            plan.bispectrum(x, B, P)
            torch.cuda.synchronize()
            one.append((B, P))
        queued = [outputs() for _ in f]
        for x, (B, P) in zip(f, queued):
            plan.bispectrum(x, B, P)
        captured = [outputs() for _ in f]
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            for x, (B, P) in zip(f, captured):
                plan.bispectrum(x, B, P)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        for a, b, c in zip(one, queued, captured):
            for k in range(2):
                assert torch.equal(a[k], b[k]) and torch.equal(a[k], c[k])
