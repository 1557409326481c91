"""What a user of the estimator has it do, as cases that can be timed and checked.

A case names one use of the library with its sizes.  ``listed()`` gives the
fixed ones, ``draw(rng)`` further ones of the same ranges, ``prepare`` builds
what a program has in hand before the call (fields on the GPU, the plan),
``run`` makes one pass through the public entry points, ``work`` counts what
the path cannot do without, and ``exact`` gives the same outputs from plain
torch in 64 bits.

The estimates are handed on in single precision, as a likelihood sampler
keeps its data vector: every transform of the path runs in FP32, so the
doubles that the C interface returns carry no more than that.
"""
import math

import numpy as np
import torch

import paper_1705_06284_gb300 as fbs
from paper_1705_06284_gb300.batch import GraphBatch

# grid sides that the library takes (even, 2^a 3^b), from the smallest in use to the largest
GRIDS = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384, 432, 486, 512]


def listed():
    return [
        # the smallest plan in use (32^3, 6 linear bins): launches and latency count
        {"name": "bispectrum_32_lin6_fp32", "use": "bispectrum", "N": 32, "bins": 6, "spacing": "lin",
         "precision": "fp32", "field": "lognormal"},
        # a sampler's request on the smallest served grid
        {"name": "bispectrum_64_lin12_bf16x3", "use": "bispectrum", "N": 64, "bins": 12, "spacing": "lin",
         "precision": "bf16x3", "field": "bubbles"},
        # a served request with the most bins (thousands of triplets, several pair tiles)
        {"name": "bispectrum_192_lin48_bf16x3", "use": "bispectrum", "N": 192, "bins": 48, "spacing": "lin",
         "precision": "bf16x3", "field": "lognormal"},
        # the toy reionisation field: FP32 transforms and FP32 products
        {"name": "bispectrum_256_lin32_fp32", "use": "bispectrum", "N": 256, "bins": 32, "spacing": "lin",
         "precision": "fp32", "field": "bubbles"},
        # the largest served grid, an odd bin count
        {"name": "bispectrum_384_lin29_bf16x3", "use": "bispectrum", "N": 384, "bins": 29, "spacing": "lin",
         "precision": "bf16x3", "field": "lognormal"},
        # the headline step: B on 64 log bins and T on 16 from one forward transform
        {"name": "both_512_log64_log16_bf16x3", "use": "both", "N": 512, "bins": 64, "bins_T": 16, "spacing": "log",
         "precision": "bf16x3", "field": "quadratic"},
        # a trispectrum in FP32 products
        {"name": "trispectrum_108_log10_fp32", "use": "trispectrum", "N": 108, "bins": 10, "spacing": "log",
         "precision": "fp32", "field": "quadratic"},
        # the connected trispectrum on a grid side without compile-time radices
        {"name": "connected_162_log9_bf16x3", "use": "connected", "N": 162, "bins": 9, "spacing": "log",
         "precision": "bf16x3", "field": "lognormal"},
        # the trispectrum resolved by the quadrilateral's diagonal
        {"name": "diagonal_96_lin6_d8_fp32", "use": "diagonal", "N": 96, "bins": 6, "diag": 8, "spacing": "lin",
         "precision": "fp32", "field": "quadratic"},
        # realisations of uneven grids replayed as one CUDA graph
        {"name": "graph_24_lin24_bf16x3", "use": "graph", "fields": 24, "bins": 24, "spacing": "lin",
         "precision": "bf16x3"},
        # many realisations of one grid in one set of launches, FP32 products
        {"name": "batch_96_x16_lin24_fp32", "use": "batch", "N": 96, "fields": 16, "bins": 24, "spacing": "lin",
         "precision": "fp32", "field": "lognormal"},
        # a complex field on a non-cubic grid
        {"name": "general_96x72x108_log8", "use": "general", "Nx": 96, "Ny": 72, "Nz": 108, "bins": 8},
    ]


def draw(rng):
    use = rng.choice(["bispectrum", "bispectrum", "bispectrum", "both", "trispectrum", "connected", "diagonal",
                      "graph", "batch", "general"])
    field = rng.choice(["lognormal", "bubbles", "quadratic"])
    precision = rng.choice(["bf16x3", "bf16x3", "fp32"])
    spacing = rng.choice(["lin", "log"])

    def grid(lo, hi):  # even over the logarithm
        x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min((g for g in GRIDS if lo <= g <= hi), key=lambda g: abs(math.log(g / x)))

    if use == "bispectrum":
        N = grid(16, 256 if precision == "fp32" else 512)
        return {"use": use, "N": N, "bins": rng.randint(4, max(5, min(N // 4, 32 if precision == "fp32" else 48))),
                "spacing": spacing, "precision": precision, "field": field}
    if use == "both":
        N = grid(64, 432)
        return {"use": use, "N": N, "bins": rng.randint(12, 64 if N > 128 else 32), "bins_T": rng.randint(6, 16),
                "spacing": "log", "precision": "bf16x3", "field": field}
    if use == "trispectrum":
        N = grid(24, 128 if precision == "fp32" else 256)
        return {"use": use, "N": N, "bins": rng.randint(4, 10 if precision == "fp32" else 16), "spacing": spacing,
                "precision": precision, "field": field}
    if use == "connected":
        return {"use": use, "N": grid(32, 216), "bins": rng.randint(4, 12), "spacing": "log", "precision": "bf16x3",
                "field": field}
    if use == "diagonal":
        return {"use": use, "N": grid(24, 108), "bins": rng.randint(4, 7), "diag": rng.randint(4, 12),
                "spacing": spacing, "precision": precision, "field": field}
    if use == "graph":
        return {"use": use, "fields": rng.randint(5, 32), "bins": rng.randint(12, 28), "spacing": "lin",
                "precision": "bf16x3"}
    if use == "batch":
        N = grid(32, 128)
        most = 20 if N > 72 else 40
        return {"use": use, "N": N, "fields": rng.randint(3, most), "bins": rng.randint(6, min(24, N // 4)),
                "spacing": spacing, "precision": precision, "field": field}
    sides = [27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128]
    return {"use": "general", "Nx": rng.choice(sides), "Ny": rng.choice(sides), "Nz": rng.choice(sides),
            "bins": rng.randint(4, 9)}


# ---------------------------------------------------------------- inputs
def _edges(N, L, bins, spacing):
    kf = 2.0 * math.pi / L  # from k_f to half the Nyquist wavenumber
    return (np.linspace if spacing == "lin" else np.geomspace)(kf, 0.25 * N * kf, bins + 1)


def _diag_edges(N, L, bins):
    kf = 2.0 * math.pi / L  # q = 0 alone, then shells up to the longest diagonal
    return np.concatenate([[0.0], np.linspace(0.5 * kf, 0.5 * N * kf, bins)])


def _side(N):
    return 1.0 * N  # cells of unit length


def _general(case):
    shape = (case["Nx"], case["Ny"], case["Nz"])
    Ls = tuple(1.0 * n * s for n, s in zip(shape, (1.0, 1.25, 0.8)))
    lo = 2 * math.pi / max(Ls)
    hi = 2 * math.pi * min(n / 4.0 / L for n, L in zip(shape, Ls))
    return shape, Ls, np.geomspace(1.2 * lo, 0.999 * hi, case["bins"] + 1)


def _gaussian(N, slope, sigma, gen):
    f = torch.fft.fftfreq(N, 1.0 / N, device="cuda")
    k2 = (f ** 2)[:, None, None] + (f ** 2)[None, :, None] + (f[: N // 2 + 1] ** 2)[None, None, :]
    k2[0, 0, 0] = 1.0
    w = torch.fft.rfftn(torch.randn((N, N, N), device="cuda", generator=gen)) * k2 ** (0.25 * slope)
    w[0, 0, 0] = 0.0
    g = torch.fft.irfftn(w, s=(N, N, N))
    return g * (sigma / g.square().mean().sqrt())


def _field(kind, N, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "bubbles":  # equal-radius spheres, overlap allowed, about half the volume
        R = max(2.0, min(6.0, N / 12.0))
        n = int(math.log(2.0) * N ** 3 / (4.0 / 3.0 * math.pi * R ** 3))
        centres = torch.randint(0, N ** 3, (n,), device="cuda", generator=gen)
        points = torch.zeros(N ** 3, device="cuda")
        points[centres] = 1.0
        d2 = torch.fft.fftfreq(N, 1.0 / N, device="cuda") ** 2
        ball = (d2[:, None, None] + d2[None, :, None] + d2[None, None, :] <= R * R).float()
        hit = torch.fft.irfftn(torch.fft.rfftn(points.view(N, N, N)) * torch.fft.rfftn(ball), s=(N, N, N))
        neutral = (hit < 0.5).float()
        return (neutral / neutral.mean() - 1.0).contiguous()
    if kind == "lognormal":
        return (torch.exp(_gaussian(N, -2.0, 0.5, gen) - 0.125) - 1.0).contiguous()
    g = _gaussian(N, -1.5, 0.1, gen)  # quadratic local
    g2 = g.square()
    return (g + 0.3 * (g2 - g2.mean())).contiguous()


def _mixed(case, seed):
    """Realisations of a mixed batch: grids of 64, 96 and 128, half lognormal, half bubbles."""
    return [_field("lognormal" if i % 2 else "bubbles", (64, 96, 128)[(i + i // 3) % 3], 1000 * seed + i)
            for i in range(case["fields"])]


def _complex_field(shape, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = torch.complex(torch.randn(shape, device="cuda", generator=gen), torch.randn(shape, device="cuda", generator=gen))
    return (g + 0.3 * g * g).contiguous()


def _input(case, seed):
    if case["use"] == "graph":
        return _mixed(case, seed)
    if case["use"] == "batch":
        return [_field(case["field"], case["N"], 1000 * seed + i) for i in range(case["fields"])]
    if case["use"] == "general":
        return _complex_field(_general(case)[0], seed)
    return _field(case["field"], case["N"], seed)


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    use, data = case["use"], _input(case, seed)
    if use == "general":
        torch.cuda.synchronize()  # the general plan works on its own stream
        return {"use": use, "plan": fbs.GeneralPlan(*_general(case)), "data": data}
    if use == "graph":
        torch.cuda.synchronize()  # the batch works on its own stream
        batch = GraphBatch(data, L_for=_side, edges_for=lambda N: _edges(N, _side(N), case["bins"], case["spacing"]),
                           precision=case["precision"], tune=False)
        batch.capture()
        return {"use": use, "batch": batch, "grids": sorted(batch.groups)}
    N, L = case["N"], _side(case["N"])
    plan = fbs.Plan(N, L, _edges(N, L, case["bins"], case["spacing"]), precision=case["precision"],
                    trispectrum=use in ("trispectrum", "connected", "diagonal"))
    state = {"use": use, "plan": plan, "data": data}
    if use == "both":
        state["plan_T"] = fbs.Plan(N, L, _edges(N, L, case["bins_T"], case["spacing"]), precision=case["precision"],
                                   trispectrum=True)
        state["plan_T"].follow(plan)
    if use == "diagonal":
        plan.set_diagonal(_diag_edges(N, L, case["diag"]))
    return state


def run(state):
    use = state["use"]
    if use == "graph":
        batch = state["batch"]
        batch.stream.wait_stream(torch.cuda.current_stream())
        batch.replay()
        torch.cuda.current_stream().wait_stream(batch.stream)
        return {str(N): [batch.groups[N]["B"].float(), batch.groups[N]["P"].float()] for N in state["grids"]}
    plan, data = state["plan"], state["data"]
    if use == "general":
        B, P = plan.bispectrum(data)
        return {"B": B.astype(np.complex64), "P": P.astype(np.complex64)}
    if use == "batch":
        B, P = plan.bispectrum_batch(data)
        return {"B": B.float(), "P": P.float()}
    if use == "both":
        B, P = plan.bispectrum(data)
        T, B_T, P_T = state["plan_T"].trispectrum(None)
        return {"B": B.float(), "P": P.float(), "T": T.float(), "B_T": B_T.float(), "P_T": P_T.float()}
    if use == "trispectrum":
        T, B, P = plan.trispectrum(data)
        return {"T": T.float(), "B": B.float(), "P": P.float()}
    if use == "connected":
        Tc, T, B, P = plan.trispectrum_connected(data)
        return {"Tc": Tc.float(), "T": T.float(), "B": B.float(), "P": P.float()}
    if use == "diagonal":
        return {"TD": plan.trispectrum_diagonal(data).float()}
    B, P = plan.bispectrum(data)
    return {"B": B.float(), "P": P.float()}


# ---------------------------------------------------------------- the closed items, from the shells alone
def _thresholds(edges, L):
    """Integers t with bin b = {t_b <= |m|^2 < t_{b+1}} (edges within 1e-9 of a lattice value are on it)."""
    out = []
    for e in edges:
        x = (e * L / (2.0 * math.pi)) ** 2
        r = round(x)
        out.append(int(r if abs(x - r) <= 1e-9 * max(1.0, x) else math.ceil(x)))
    return out


def _reach(thr, top):
    """(smallest, largest) |m| that occurs in each bin, or None for an empty one."""
    sums = {x * x + y * y for x in range(top + 1) for y in range(x, top + 1)}
    occurs = sorted({s + z * z for s in sums for z in range(top + 1) if s + z * z < thr[-1]})
    out = []
    for lo, hi in zip(thr, thr[1:]):
        s = [v for v in occurs if lo <= v < hi]
        out.append((math.sqrt(s[0]), math.sqrt(s[-1])) if s else None)
    return out


def _closing(reach, arity):
    """Bin tuples in ascending order whose shells can close a polygon."""
    have = [b for b, r in enumerate(reach) if r]

    def extend(head):
        if len(head) == arity:
            if reach[head[-1]][0] <= sum(reach[b][1] for b in head[:-1]) + 1e-9:
                yield tuple(head)
            return
        for b in have:
            if not head or b >= head[-1]:
                yield from extend(head + [b])

    return list(extend([]))


def _grid(need, N):
    """Smallest side above `need` of the form 2^a 3^b, at most N."""
    good = [n for n in range(8, N + 1, 2) if n == 2 ** round(math.log2(n & -n)) * 3 ** round(math.log(n // (n & -n), 3))]
    return next((n for n in good if n > need), N)


def work(case):
    use = case["use"]
    if use == "general":
        shape, Ls, edges = _general(case)
        n, nb = float(np.prod(shape)), case["bins"]
        items = nb * (nb + 1) * (nb + 2) / 6
        return {"bytes": 8 * n + 16 * (items + nb), "flops": 5 * n * math.log2(n) * (1 + nb) + 8 * items * n}

    def one(N, bins, spacing, arities, forward=True):
        thr = _thresholds(_edges(N, _side(N), bins, spacing), _side(N))
        top = math.isqrt(thr[-1])
        reach = _reach(thr, top)
        R = [math.isqrt(t - 1) for t in thr[1:]]
        flops, largest, out = 2.5 * N ** 3 * math.log2(N ** 3) if forward else 0.0, {}, bins
        for arity in arities:
            for item in _closing(reach, arity):
                M = _grid(max(sum(R[b] for b in item), 2 * R[item[-1]]), N)
                flops += 2.0 * M ** 3
                out += 1
                for b in item:
                    largest[b] = max(largest.get(b, 0), M)
        flops += sum(2.5 * M ** 3 * math.log2(M ** 3) for M in largest.values())  # each shell field once
        return {"bytes": (4.0 * N ** 3 if forward else 0.0) + 4.0 * out, "flops": flops}

    if use == "graph":
        parts = []
        for i in range(case["fields"]):
            parts.append((64, 96, 128)[(i + i // 3) % 3])
        each = {N: one(N, case["bins"], case["spacing"], (3,)) for N in set(parts)}
        return {k: sum(each[N][k] for N in parts) for k in ("bytes", "flops")}
    quads = use in ("trispectrum", "connected", "diagonal")
    w = one(case["N"], case["bins"], case["spacing"], (4,) if use == "diagonal" else (3, 4) if quads else (3,))
    if use == "both":
        t = one(case["N"], case["bins_T"], case["spacing"], (3, 4), forward=False)
        w = {k: w[k] + t[k] for k in w}
    if use == "batch":
        w = {k: v * case["fields"] for k, v in w.items()}
    return w


# ---------------------------------------------------------------- the same outputs in 64 bits
class _Shells:
    """Shell fields of a real cubic field (or of the indicator, field None) on the smallest grid that keeps `p`-fold sums."""

    def __init__(self, N, thr, p, field):
        dev = torch.device("cuda")
        R = math.isqrt(thr[-1] - 1)
        self.N, self.M = N, _grid(p * R, N)
        M = self.M
        m = torch.arange(-R, R + 1, device=dev)
        mz = torch.arange(0, R + 1, device=dev)
        self.m2 = (m * m)[:, None, None] + (m * m)[None, :, None] + (mz * mz)[None, None, :]
        if field is None:
            self.D = torch.ones(self.m2.shape, device=dev, dtype=torch.complex128)
        else:
            D = torch.fft.rfftn(field.double())
            self.D = D.index_select(0, m % N).index_select(1, m % N)[:, :, : R + 1].contiguous()
        self.weight = torch.where(mz == 0, 1.0, 2.0).double()  # m and -m, of which the box holds mz >= 0
        self.shells = [(self.m2 >= lo) & (self.m2 < hi) for lo, hi in zip(thr, thr[1:])]
        self.fields = torch.zeros((len(self.shells), M ** 3), device=dev, dtype=torch.float64)
        box = torch.zeros((M, M, M // 2 + 1), device=dev, dtype=torch.complex128)
        for b, s in enumerate(self.shells):
            box.zero_()
            part = torch.where(s, self.D, torch.zeros_like(self.D))
            box[(m % M)[:, None], (m % M)[None, :], : R + 1] = part
            self.fields[b] = (torch.fft.irfftn(box, s=(M, M, M)) * float(M) ** 3).reshape(-1)

    def moment(self, b, power):
        return float((self.D.abs() ** power * self.weight * self.shells[b]).sum())

    def sums(self, items):
        """sum over the N^3 grid of each item's product, divided by N^3: a tensor in the order of `items`."""
        F, out, i = self.fields, [], 0
        have = {}
        for it in items:  # items of the same tail share its product
            have.setdefault(it[1:], []).append(it[0])
        for tail, heads in have.items():
            prod = F[tail[0]]
            for b in tail[1:]:
                prod = prod * F[b]
            lo, hi = min(heads), max(heads)
            v = torch.mv(F[lo:hi + 1], prod).cpu()
            out += [((a,) + tail, float(v[a - lo]) / self.M ** 3) for a in heads]
        got = dict(out)
        return torch.tensor([got[it] for it in items], dtype=torch.float64)


def _cubic(field, N, bins, spacing, arities):
    """(fields' shells, the indicator's, {arity: (items, sums, counts)}, P) of a real cubic field."""
    L = _side(N)
    thr = _thresholds(_edges(N, L, bins, spacing), L)
    reach = _reach(thr, math.isqrt(thr[-1]))
    cand = {a: _closing(reach, a) for a in arities}
    ones = _Shells(N, thr, max(arities), None)
    counts = {a: torch.round(ones.sums(cand[a])) for a in arities}
    size = torch.tensor([ones.moment(b, 0) for b in range(bins)], dtype=torch.float64)
    del ones.fields
    data = _Shells(N, thr, max(arities), field)
    got = {}
    for a in arities:
        keep = counts[a] > 0
        items = [it for it, k in zip(cand[a], keep.tolist()) if k]
        got[a] = (items, data.sums(items), counts[a][keep])
    power = torch.tensor([data.moment(b, 2) for b in range(bins)], dtype=torch.float64)
    V, n = L ** 3, float(N) ** 3
    P = V / n ** 2 * power / size  # an empty bin: 0/0
    return data, thr, got, P, size


def _estimate(N, arity, sums, counts):
    V, n = _side(N) ** 3, float(N) ** 3
    return V ** (arity - 1) / n ** arity * sums / counts


def _exact_B(field, N, bins, spacing):
    data, thr, got, P, size = _cubic(field, N, bins, spacing, (3,))
    return _estimate(N, 3, *got[3][1:]), P


def _exact_T(field, N, bins, spacing, connected=False):
    data, thr, got, P, size = _cubic(field, N, bins, spacing, (3, 4))
    items, sums, counts = got[4]
    T, B = _estimate(N, 4, sums, counts), _estimate(N, 3, *got[3][1:])
    if not connected:
        return T, B, P
    # leave out the quadruples with two modes that cancel (no bin holds a self-conjugate mode)
    paired, n_paired = torch.zeros_like(sums), torch.zeros_like(counts)
    for i, (a, b, c, d) in enumerate(items):
        if a == b and c == d:
            s2 = data.moment(a, 2)
            paired[i] = 3 * s2 * s2 - 3 * data.moment(a, 4) if a == c else s2 * data.moment(c, 2)
            n_paired[i] = 3 * size[a] ** 2 - 3 * size[a] if a == c else size[a] * size[c]
    left = torch.round(counts - n_paired)
    Tc = _estimate(N, 4, sums - paired, left)
    return torch.where(left > 0, Tc, torch.full_like(Tc, float("nan"))), T, B, P


def _exact_diagonal(field, case):
    N, L = case["N"], _side(case["N"])
    data, thr, got, P, size = _cubic(field, N, case["bins"], case["spacing"], (4,))
    items = got[4][0]
    ones = _Shells(N, thr, 4, None)
    M = data.M
    q = torch.fft.fftfreq(M, 1.0 / M, device="cuda").double().round()
    q2 = (q * q)[:, None, None] + (q * q)[None, :, None] + (q * q)[None, None, :]
    dthr = _thresholds(_diag_edges(N, L, case["diag"]), L)
    shells = [((q2 >= lo) & (q2 < hi)).reshape(-1).nonzero().reshape(-1) for lo, hi in zip(dthr, dthr[1:])]
    out = torch.zeros((len(items), len(shells)), dtype=torch.float64)
    sides = []
    for s in (data, ones):
        pairs = {p for it in items for p in (it[:2], it[2:])}
        spec = {p: torch.fft.fftn((s.fields[p[0]] * s.fields[p[1]]).view(M, M, M)).reshape(-1) / M ** 3 for p in pairs}
        v = torch.zeros((len(items), len(shells)), dtype=torch.float64)
        for i, it in enumerate(items):
            g = (spec[it[:2]] * spec[it[2:]].conj()).real
            for d, idx in enumerate(shells):
                v[i, d] = float(g[idx].sum())
        sides.append(v)
    num, cnt = sides[0], torch.round(sides[1])
    out = _estimate(N, 4, num, cnt)
    return torch.where(cnt > 0, out, torch.full_like(out, float("nan")))


def _exact_general(case, field):
    shape, Ls, edges = _general(case)
    nb, n, V = case["bins"], float(np.prod(shape)), float(np.prod(Ls))
    t = torch.tensor([(e / (2.0 * math.pi)) ** 2 for e in edges], dtype=torch.float64, device="cuda")
    u = [(torch.fft.fftfreq(k, 1.0 / k, device="cuda", dtype=torch.float64).round() / L) for k, L in zip(shape, Ls)]
    s = ((u[0] * u[0])[:, None, None] + (u[1] * u[1])[None, :, None]) + (u[2] * u[2])[None, None, :]
    which = torch.bucketize(s, t, right=True) - 1
    D = torch.fft.fftn(field.to(torch.complex128))
    masks = [which == b for b in range(nb)]
    size = [int(m.sum()) for m in masks]
    I = [torch.fft.ifftn(torch.where(m, D, torch.zeros_like(D))).reshape(-1) * n for m in masks]
    C = [torch.fft.ifftn(m.to(torch.complex128)).real.reshape(-1) * n for m in masks]
    B = []
    for a in range(nb):
        for b in range(a, nb):
            for c in range(b, nb):
                if not (size[a] and size[b] and size[c]):
                    continue
                cnt = round(float((C[a] * C[b] * C[c]).sum()) / n)
                if cnt > 0:
                    B.append(complex((I[a] * I[b] * I[c]).sum()) * V ** 2 / n ** 3 / (n * cnt))
    P = [complex((I[b] * I[b]).sum()) * V / n ** 2 / (n * size[b]) if size[b] else complex("nan+nanj")
         for b in range(nb)]
    return np.array(B, dtype=np.complex128), np.array(P, dtype=np.complex128)


def exact(case, seed):
    use, data = case["use"], _input(case, seed)
    if use == "general":
        B, P = _exact_general(case, data)
        return {"B": B, "P": P}
    if use == "graph":
        got = {}
        for f in data:
            N = f.shape[0]
            got.setdefault(N, []).append(_exact_B(f, N, case["bins"], case["spacing"]))
        return {str(N): [torch.stack([x[0] for x in v]), torch.stack([x[1] for x in v])] for N, v in got.items()}
    N, bins, spacing = case["N"], case["bins"], case["spacing"]
    if use == "batch":
        v = [_exact_B(f, N, bins, spacing) for f in data]
        return {"B": torch.stack([x[0] for x in v]), "P": torch.stack([x[1] for x in v])}
    if use == "diagonal":
        return {"TD": _exact_diagonal(data, case)}
    if use == "trispectrum":
        T, B, P = _exact_T(data, N, bins, spacing)
        return {"T": T, "B": B, "P": P}
    if use == "connected":
        Tc, T, B, P = _exact_T(data, N, bins, spacing, connected=True)
        return {"Tc": Tc, "T": T, "B": B, "P": P}
    B, P = _exact_B(data, N, bins, spacing)
    if use != "both":
        return {"B": B, "P": P}
    T, B_T, P_T = _exact_T(data, N, case["bins_T"], spacing)
    return {"B": B, "P": P, "T": T, "B_T": B_T, "P_T": P_T}
