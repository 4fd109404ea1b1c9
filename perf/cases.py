"""The work that users of this library have it do, as cases that can be timed and compared.

Four kinds of call, each through the public binding:

  op      one application of the Galerkin operator, ``Context.matvec`` -- the call a user's own
          Krylov solver makes, and what every solve below consists of (FP64 and FP32, primal and
          dual, d = 2 and 3, cubic and ragged orders)
  bounds  a whole bound pair, ``Context.bounds`` (both precisions, disks, squares and spheres)
  batch   many small microstructures solved together, ``Batch.submit / run / results``
  setup   a new microstructure in an existing context, ``Context.set_coeffs``, and its data back
          (``table`` and ``grid_values``)

Sizes are those of the tests, the benchmark and the request streams in ``workloads``: d = 2 orders
15 .. 2187, d = 3 orders 15 .. 129, batches of disks with orders 31 .. 255.
"""
import math

import numpy as np
import torch

import paper_1412_2033_gb300 as g

BOX, DISK, SPHERE = 0, 1, 2


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _op(name, N, prec, kind, shape, count, contrast):
    n = list(N) + [0] * (3 - len(N))
    c = {"call": "op", "d": len(N), "N0": n[0], "N1": n[1], "N2": n[2], "prec": prec, "kind": kind, "shape": shape,
         "count": count, "contrast": contrast}
    return dict(c, name=name) if name else c


def _bounds(name, d, N, prec, shape, count, contrast):
    c = {"call": "bounds", "d": d, "N0": N, "N1": N, "N2": N if d == 3 else 0, "prec": prec, "shape": shape,
         "count": count, "contrast": contrast}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one operator application in a user's solver on a small cell: a handful of microseconds of
        # launches (the order of the smallest served 2-D request)
        _op("op_f32_2d_n63", (63, 63), "f32", "primal", "disk", 5, 100.0),
        # an odd, ragged 2-D order out of the served range, in the default precision
        _op("op_f64_2d_n315x517", (315, 517), "f64", "dual", "disk", 10, 50.0),
        # the largest served 2-D order: its double grid 2048 is a power of two
        _op("op_f32_2d_n1023", (1023, 1023), "f32", "primal", "disk", 20, 1000.0),
        # the benchmark's 2-D order, both precisions: the inner iteration and the residual correction
        _op("op_f32_2d_n2187", (2187, 2187), "f32", "dual", "disk", 1, 100.0),
        _op("op_f64_2d_n2187", (2187, 2187), "f64", "primal", "disk", 1, 100.0),
        # d = 3: the largest order in FP32, a ragged one in FP64
        _op("op_f32_3d_n129", (129, 129, 129), "f32", "primal", "sphere", 1, 1000.0),
        _op("op_f64_3d_n63x99x77", (63, 99, 77), "f64", "primal", "sphere", 4, 100.0),
        # whole bound pairs: the benchmark's, a d = 3 one, and a small one in the default precision
        _bounds("bounds_mixed_2d_n2187", 2, 2187, "mixed", "disk", 1, 100.0),
        _bounds("bounds_mixed_3d_n65", 3, 65, "mixed", "sphere", 1, 1000.0),
        _bounds("bounds_f64_2d_n81", 2, 81, "fp64", "box", 1, 10.0),
        # many microstructures at once, orders and contrasts as they come
        {"name": "batch_2d_64", "call": "batch", "count": 64, "lo": 31, "hi": 255},
        # the next microstructure of a parameter study in the same context
        {"name": "setup_2d_n1023", "call": "setup", "d": 2, "N0": 1023, "N1": 1023, "N2": 0, "shape": "disk",
         "count": 20, "contrast": 1000.0},
    ]


def _odd(rng, lo, hi):
    """An odd number in lo .. hi (both odd), uniform in its logarithm."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))
    return min(hi, max(lo, n | 1))


def draw(rng):
    call = rng.choice(["op"] * 5 + ["bounds"] * 3 + ["batch", "setup"])
    contrast = round(math.exp(rng.uniform(math.log(2.0), math.log(1000.0))), 3)
    d = rng.choice([2, 3])
    shape = rng.choice(["box", "disk" if d == 2 else "sphere"])
    count = 1 if shape == "box" else rng.randint(1, 20 if d == 2 else 8)
    if call == "op":
        if d == 2:
            N = (_odd(rng, 15, 2187), _odd(rng, 15, 2187))
            N = rng.choice([N, (N[0], N[0])])
        else:
            N = tuple(_odd(rng, 15, 129) for _ in range(3))
            N = rng.choice([N, (N[0],) * 3])
        return _op(None, N, rng.choice(["f32", "f64"]), rng.choice(["primal", "dual"]), shape, count, contrast)
    if call == "bounds":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        N = _odd(rng, 15, (1215 if prec == "mixed" else 405)) if d == 2 else _odd(rng, 15, (65 if prec == "mixed" else 33))
        return _bounds(None, d, N, prec, shape, count, min(contrast, 300.0))
    if call == "batch":
        return {"call": "batch", "count": int(math.exp(rng.uniform(math.log(4), math.log(64)))), "lo": 31,
                "hi": _odd(rng, 63, 255)}
    N = _odd(rng, 15, 1023) if d == 2 else _odd(rng, 15, 99)
    return {"call": "setup", "d": d, "N0": N, "N1": N, "N2": N if d == 3 else 0, "shape": shape, "count": count,
            "contrast": contrast}


def _orders(case):
    return [case["N0"], case["N1"], case["N2"]][: case["d"]]


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _inclusions(r, d, shape, count, contrast):
    """A fraction of the cell in inclusions of the given contrast: one box or ball of the benchmark's
    size (about 0.2 .. 0.3 of the cell) anywhere in it, or several disjoint smaller balls."""
    if shape == "box":
        side = r.uniform(0.55, 0.7, size=d)
        return [(BOX, tuple(r.uniform(-0.5, 0.5, size=d)), tuple(side), contrast)]
    kind = DISK if d == 2 else SPHERE
    if count == 1:
        f = r.uniform(0.28, 0.32) if d == 2 else r.uniform(0.18, 0.22)
        rad = math.sqrt(f / math.pi) if d == 2 else (3 * f / (4 * math.pi)) ** (1 / 3)
        return [(kind, tuple(r.uniform(-0.5, 0.5, size=d)), (rad,), contrast)]
    lo, hi = (0.03, 0.12) if d == 2 else (0.05, 0.2)
    placed = []
    for _ in range(20000):
        if len(placed) == count:
            break
        rad, c = r.uniform(lo, hi), r.uniform(-0.5, 0.5, size=d)
        if all(np.linalg.norm((c - q) - np.round(c - q)) > 1.001 * (rad + s) for q, s in placed):
            placed.append((c, rad))
    return [(kind, tuple(float(v) for v in c), (float(s),), contrast) for c, s in placed]


def _micro(case, seed):
    return _inclusions(np.random.default_rng(seed), case["d"], case["shape"], case["count"], case["contrast"])


def _field(N, dtype, seed):
    """A trial field as a solver holds it: a real trigonometric polynomial whose coefficients fall off
    like 1/(1 + |k|) (half spectrum, Hermitian on the plane k_d = 0)."""
    d, h = len(N), (N[-1] + 1) // 2
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((d, *N[:-1], h), dtype=torch.complex128, device="cuda", generator=gen)
    k2 = sum(k * k for k in _freq(N))
    x = x / (1.0 + k2.sqrt())
    axes = tuple(range(1, d))
    x[..., 0] = 0.5 * (x[..., 0] + x[..., 0].flip(axes).conj())
    return x.to(dtype).contiguous()


def _freq(N):
    """The frequencies of a half spectrum, one broadcastable tensor per axis (k_d >= 0 on the last)."""
    d = len(N)
    out = []
    for a, n in enumerate(N):
        k = torch.arange((n + 1) // 2, device="cuda") if a == d - 1 else torch.arange(n, device="cuda") - (n - 1) // 2
        out.append(k.double().reshape([-1 if b == a else 1 for b in range(d)]))
    return out


def _batch(case, seed):
    r = np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        n = int(2 * r.integers((case["lo"] - 1) // 2, (case["hi"] - 1) // 2 + 1) + 1)
        contrast = float(np.exp(r.uniform(math.log(2.0), math.log(1e4))))
        out.append({"d": 2, "N": [n, n], "a0": 1.0,
                    "inclusions": _inclusions(r, 2, "disk", int(r.integers(2, 21)), contrast)})
    return out


def prepare(case, seed):
    if case["call"] == "batch":
        return {"call": "batch", "batch": g.Batch(), "micros": _batch(case, seed)}
    d, N, inc = case["d"], _orders(case), _micro(case, seed)
    if case["call"] == "setup":
        # the context comes from the study's previous microstructure
        before = _inclusions(np.random.default_rng(seed + 1), d, "box", 1, 2.0)
        return {"call": "setup", "ctx": g.Context(d, N, 1.0, before), "inc": inc}
    if case["call"] == "bounds":
        return {"call": "bounds", "ctx": g.Context(d, N, 1.0, inc, precision=case["prec"])}
    dtype = torch.complex64 if case["prec"] == "f32" else torch.complex128
    return {"call": "op", "ctx": g.Context(d, N, 1.0, inc), "x": _field(N, dtype, seed),
            "kind": g.GHB_PRIMAL if case["kind"] == "primal" else g.GHB_DUAL}


def run(state):
    if state["call"] == "op":
        return {"y": state["ctx"].matvec(state["x"], kind=state["kind"])}
    if state["call"] == "bounds":
        upper, lower, _, status = state["ctx"].bounds()
        return {"upper": upper, "lower": lower, "status": status}
    if state["call"] == "batch":
        b = state["batch"]
        for m in state["micros"]:
            b.submit(m)
        b.run()
        res = sorted(b.results(), key=lambda r: r["id"])
        return {"upper": np.stack([r["upper"] for r in res]), "lower": np.stack([r["lower"] for r in res]),
                "status": np.array([r["status"] for r in res], dtype=np.int64)}
    ctx = state["ctx"]
    ctx.set_coeffs(1.0, state["inc"])
    return {"table": ctx.table(g.GHB_PRIMAL), "inverse_table": ctx.table(g.GHB_DUAL),
            "grid": ctx.grid_values(g.GHB_PRIMAL), "inverse_grid": ctx.grid_values(g.GHB_DUAL)}


# ------------------------------------------------------------------------------------------------
# work and the values in 64 bits
# ------------------------------------------------------------------------------------------------
def _pairs(N):
    """(entries of one component's half spectrum, points of the smallest double grid)."""
    return math.prod(N[:-1]) * ((N[-1] + 1) // 2), math.prod(2 * n - 1 for n in N)


def _operator_flops(N):
    """Real transforms there and back on the double grid, 2.5 L log2 L each per component."""
    pts = _pairs(N)[1]
    return 2 * len(N) * 2.5 * pts * math.log2(max(pts, 2))


def _iterations(contrast, tol=1e-10):
    """What conjugate gradients take at most for this contrast (their classical bound)."""
    return math.ceil(0.5 * math.sqrt(contrast) * math.log(2 / tol))


def work(case):
    if case["call"] == "batch":
        n = [i for i in range(case["lo"], case["hi"] + 1, 2)]
        flops = sum(4 * _iterations(140.0) * _operator_flops([i, i]) for i in n) / len(n)
        data = sum(2 * 4 * _pairs([i, i])[1] for i in n) / len(n)
        return {"bytes": case["count"] * data, "flops": case["count"] * flops}
    N = _orders(case)
    d = len(N)
    field, grid = _pairs(N)
    if case["call"] == "op":
        e = 8 if case["prec"] == "f32" else 16
        return {"bytes": 2 * d * field * e + grid * e / 2, "flops": _operator_flops(N)}
    if case["call"] == "bounds":
        return {"bytes": 2 * grid * (4 if case["prec"] == "mixed" else 8),
                "flops": 2 * d * _iterations(case["contrast"]) * _operator_flops(N)}
    table = math.prod(2 * n - 1 for n in N[:-1]) * N[-1]
    return {"bytes": 2 * (16 * table + 8 * grid), "flops": 2 * 2.5 * grid * math.log2(max(grid, 2)) + 40.0 * table * case["count"]}


def _smooth(n):
    """The smallest m >= n with prime factors 2, 3 and 5: the double grid that a context takes for n = 2N - 1."""
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _j1(x):
    """The Bessel function J_1 (x >= 0) in 64 bits: the trapezoidal rule on its integral (1/2 pi) int cos(t - x sin t) dt,
    which converges geometrically, up to x = 25, and Hankel's asymptotic expansion (Abramowitz and Stegun 9.2.5) above."""
    big = x.clamp(min=25.0)
    p, q, a = torch.ones_like(x), torch.zeros_like(x), torch.ones_like(x)
    for m in range(1, 31):
        a = a * ((4.0 - (2 * m - 1) ** 2) / (8.0 * m)) / big
        s = -1.0 if (m // 2) % 2 else 1.0
        if m % 2:
            q = q + s * a
        else:
            p = p + s * a
    out = (2 / (math.pi * big)).sqrt() * (p * (big.sin() - big.cos()) + q * (big.sin() + big.cos())) / math.sqrt(2.0)
    low = x < 25.0
    v, total = x[low], 0.0
    for i in range(128):
        t = 2 * math.pi * i / 128
        total = total + torch.cos(t - v * math.sin(t))
    out[low] = total / 128
    return out


def _table(N, inc, dual):
    """Fourier coefficients of a (or 1/a), a = 1 plus inclusions, on the half of Z_{2N-1}."""
    k = _freq([2 * n - 1 for n in N])
    rho = sum(v * v for v in k).sqrt()
    t = torch.zeros(rho.shape, dtype=torch.complex128, device="cuda")
    t[tuple(n - 1 for n in N[:-1]) + (0,)] = 1.0
    for shape, center, size, value in inc:
        jump = (1.0 / value if dual else value) - 1.0
        if shape == BOX:
            f = torch.ones_like(rho)
            for v, s in zip(k, size):
                f = f * s * torch.sinc(s * v)
        elif shape == DISK:
            q = 2 * math.pi * size[0] * rho
            f = torch.where(rho == 0, math.pi * size[0] ** 2,
                            size[0] * _j1(q) / torch.where(rho == 0, 1.0, rho))
        else:
            q = 2 * math.pi * size[0] * rho
            small = 4 / 3 * math.pi * size[0] ** 3 * (1 - q**2 / 10 + q**4 / 280 - q**6 / 15120)
            f = torch.where(q < 1e-2, small, (q.sin() - q * q.cos()) / torch.where(rho == 0, 1.0, 2 * math.pi**2 * rho**3))
        ph = sum(v * c for v, c in zip(k, center))
        ph = ph - ph.round()
        t = t + jump * f * torch.polar(torch.ones_like(ph), -2 * math.pi * ph)
    return t


def _pad(x, M):
    """A centred half spectrum (leading axes kept) zero-padded to the wrapped half spectrum of the grid M."""
    d = len(M)
    lead = x.shape[: x.dim() - d]
    out = torch.zeros((*lead, *M[:-1], M[-1] // 2 + 1), dtype=x.dtype, device=x.device)
    idx = [torch.remainder(torch.arange(n, device="cuda") - (n - 1) // 2, m) for n, m in zip(x.shape[len(lead):-1], M)]
    sel = torch.meshgrid(*idx, indexing="ij")
    out[(..., *sel, slice(0, x.shape[-1]))] = x
    return out


def _values(x, M):
    d = len(M)
    return torch.fft.irfftn(_pad(x, M), s=M, dim=tuple(range(-d, 0)), norm="forward")


def _coefficients(w, N):
    d = len(N)
    M = w.shape[-d:]
    f = torch.fft.rfftn(w, dim=tuple(range(-d, 0)), norm="forward")
    idx = [torch.remainder(torch.arange(n, device="cuda") - (n - 1) // 2, m) for n, m in zip(N[:-1], M)]
    sel = torch.meshgrid(*idx, indexing="ij")
    return f[(..., *sel, slice(0, (N[-1] + 1) // 2))]


def _project(w, N, dual):
    """G_E = k k^T / k.k (components on axis -d-1) or G_J = I - G_E, zero at k = 0."""
    d = len(N)
    k = torch.stack([v.expand(*N[:-1], (N[-1] + 1) // 2) for v in _freq(N)])
    kk = (k * k).sum(0)
    kk = torch.where(kk == 0, 1.0, kk)
    p = k * ((k * w).sum(-d - 1, keepdim=True) / kk)
    if dual:
        p = w - p
        p[(..., slice(None), *[(n - 1) // 2 for n in N[:-1]], 0)] = 0
    return p


def _dot(u, v):
    """Inner products over Z_N of half spectra with a leading batch axis."""
    t = (u * v.conj()).real
    t = t.flatten(1, -2).sum(1)
    return t[:, 0] + 2 * t[:, 1:].sum(1)


def _bound(N, inc, dual):
    """The Gram matrix of the minimisers for the unit loads, by plain conjugate gradients."""
    d = len(N)
    M = [_smooth(2 * n - 1) for n in N]
    a = _values(_table(N, inc, dual), M)
    apply = lambda x: _coefficients(a * _values(x, M), N)  # noqa: E731
    E = torch.zeros((d, d, *N[:-1], (N[-1] + 1) // 2), dtype=torch.complex128, device="cuda")
    for i in range(d):
        E[(i, i, *[(n - 1) // 2 for n in N[:-1]], 0)] = 1.0
    r = -_project(apply(E), N, dual)
    x, p = torch.zeros_like(r), r.clone()
    rr = _dot(r, r)
    bb = rr.clone()
    one = [-1] + [1] * (d + 1)
    for _ in range(3000):
        if bool((rr <= 1e-23 * bb).all()):
            break
        q = _project(apply(p), N, dual)
        al = (rr / _dot(p, q)).nan_to_num(0.0)
        x = x + al.reshape(one) * p
        r = r - al.reshape(one) * q
        new = _dot(r, r)
        p = r + (new / rr).nan_to_num(0.0).reshape(one) * p
        rr = new
    v = _values(_project(x, N, dual) + E, M).flatten(2)
    av = (a.flatten() * v).flatten(1)
    out = (av @ v.flatten(1).T / a.numel()).cpu().numpy()
    return 0.5 * (out + out.T)


def exact(case, seed):
    if case["call"] == "batch":
        return None  # hundreds of solves
    N, inc = _orders(case), _micro(case, seed)
    if case["call"] == "setup":
        M = [_smooth(2 * n - 1) for n in N]
        t = [_table(N, inc, dual) for dual in (False, True)]
        return {"table": t[0], "inverse_table": t[1], "grid": _values(t[0], M), "inverse_grid": _values(t[1], M)}
    if case["call"] == "bounds":
        return {"upper": _bound(N, inc, False), "lower": np.linalg.inv(_bound(N, inc, True)), "status": None}
    dual = case["kind"] == "dual"
    dtype = torch.complex64 if case["prec"] == "f32" else torch.complex128
    x = _field(N, dtype, seed).to(torch.complex128)
    M = [_smooth(2 * n - 1) for n in N]
    a = _values(_table(N, inc, dual), M)
    return {"y": _project(_coefficients(a * _values(x, M), N), N, dual)}
