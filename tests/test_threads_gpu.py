"""Different plans from different host threads: evaluations that launch the same
kernels with shared-memory sizes of their own, at the same time, give what each
plan gives alone (fbs.h: calls on one plan are serialised by the caller,
different plans may be used from different threads)."""
import threading

import numpy as np
import pytest
import torch

import fields
import paper_1705_06284_gb300 as fbs

pytestmark = pytest.mark.gpu


def _cubic(N, tops, precision, use="bispectrum", nb=4, **kw):
    """One plan per top edge (in k_f); each call evaluates one field n times."""
    L = float(N)
    kf = 2 * np.pi / L
    out = []
    for i, top in enumerate(tops):
        s = torch.cuda.Stream()
        p = fbs.Plan(N, L, np.linspace(kf, top * kf, nb + 1), precision=precision, stream=s.cuda_stream,
                     trispectrum=use == "diagonal", **kw)
        f = torch.from_numpy(fields.lognormal(N, 0.5, -1.5, seed=70 + i).astype(np.float32)).cuda()
        torch.cuda.synchronize()
        if use == "diagonal":
            p.set_diagonal(np.linspace(0.5 * kf, 0.4 * N * kf, 5))
            TD = torch.zeros(p.nquad * 4, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()

            def call(n, p=p, f=f, s=s, TD=TD):
                for _ in range(n):
                    p.trispectrum_diagonal(f, TD)
                s.synchronize()
                return [TD.cpu().numpy()]
        else:
            B = torch.zeros(p.ntrip, dtype=torch.float64, device="cuda")
            P = torch.zeros(p.nbins, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()

            def call(n, p=p, f=f, s=s, B=B, P=P):
                for _ in range(n):
                    p.bispectrum(f, B, P)
                s.synchronize()
                return [B.cpu().numpy(), P.cpu().numpy()]
        out.append(call)
    return out


def _general(shapes):
    rng = np.random.default_rng(5)
    out = []
    for n in shapes:
        k = 2 * np.pi / min(n)
        p = fbs.GeneralPlan(n, tuple(float(v) for v in n), np.linspace(k, 0.24 * min(n) * k, 4))
        f = rng.standard_normal(n).astype(np.float32)

        def call(n, p=p, f=f):
            for _ in range(n):
                out = p.bispectrum(f)
            return list(out)
        out.append(call)
    return out


CASES = {
    "z stage": lambda: _cubic(64, (16, 3), "fp32", nb=2, full_grid=True),
    "fp32 sums": lambda: _cubic(64, (16, 5), "fp32", nb=14),
    "bf16x3 sums": lambda: _cubic(64, (16, 7), "bf16x3", nb=12),
    "diagonal": lambda: _cubic(24, (6, 4), "fp32", use="diagonal"),
    "general": lambda: _general(((512, 16, 16), (16, 256, 16))),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_two_threads(name):
    calls = CASES[name]()
    alone = [c(1) for c in calls]
    failed = []

    def work(call, ref):
        try:
            for _ in range(10):
                got = call(300)
                if not all(np.array_equal(a, b, equal_nan=True) for a, b in zip(got, ref)):
                    failed.append("outputs differ")
                    return
        except Exception as e:  # a refused launch
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=(c, r)) for c, r in zip(calls, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
