"""Evaluations captured without a warm-up of their own: tables that a call finds
missing are built beside the capture, whichever call came before it."""
import numpy as np
import pytest
import torch

import fields
import paper_1705_06284_gb300 as fbs

pytestmark = pytest.mark.gpu

N, L = 64, 64.0


def _plan(stream, precision, trispectrum=True, nb=6):
    return fbs.Plan(N, L, fields.log_edges(N, L, nb), precision=precision, trispectrum=trispectrum,
                    stream=stream.cuda_stream)


def _outputs(*n):
    return [torch.zeros(k, dtype=torch.float64, device="cuda") for k in n]


def _captured(stream, call, mode="relaxed"):
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode=mode):
        call()
    graph.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("nb", [6, 16])
@pytest.mark.parametrize("first,then", [("trispectrum_connected", "trispectrum"),
                                        ("trispectrum", "trispectrum_connected"),
                                        ("trispectrum", "bispectrum"), ("trispectrum_connected", "bispectrum")])
def test_one_call_warms_the_other(first, then, nb):
    stream = torch.cuda.Stream()
    f = torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=90).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), _plan(stream, "bf16x3", nb=nb) as plan:
        size = {"trispectrum_connected": (plan.nquad, plan.nquad, plan.ntrip, plan.nbins),
                "trispectrum": (plan.nquad, plan.ntrip, plan.nbins), "bispectrum": (plan.ntrip, plan.nbins)}
        getattr(plan, first)(f, *_outputs(*size[first]))
        got, ref = _outputs(*size[then]), _outputs(*size[then])
        _captured(stream, lambda: getattr(plan, then)(f, *got))
        getattr(plan, then)(f, *ref)
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


@pytest.mark.parametrize("mode", ["relaxed", "thread_local", "global"])
@pytest.mark.parametrize("precision,later", [("bf16x3", "bf16x3"), ("fp32", "fp32"), ("bf16x3", "fp32"),
                                             ("fp32", "bf16x3"), ("bf16", "bf16")])
def test_first_bispectrum_captured(precision, later, mode):
    """A fresh plan, its precision changed inside the capture or not."""
    stream = torch.cuda.Stream()
    f = torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=91).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), _plan(stream, precision, trispectrum=False) as plan:
        got, ref = _outputs(plan.ntrip, plan.nbins), _outputs(plan.ntrip, plan.nbins)

        def call():
            if later != precision:
                plan.set_precision(later)
            plan.bispectrum(f, *got)
        _captured(stream, call, mode)
        plan.bispectrum(f, *ref)
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert torch.equal(a, b)
