"""The FP32 operator on the run-time plans (csrc/fft_rt.cuh) where it can go
wrong: every group size, prime stages, one pass and many, forced tiles and rows."""
import math

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -23


@pytest.fixture(scope="module")
def ghb():
    import paper_1412_2033_gb300 as g
    g.load_library()
    return g


# double grids: groups of 2 .. 16 entries, padded and not, primes 7 .. 31, no pass, one pass, many
# passes, and enough warps for the kernels of 64 registers
GRIDS = [((1, 1), (1, 1)), ((1, 3), (1, 5)), ((3, 5), (8, 9)), ((7, 7), (15, 16)), ((13, 15), (25, 31)), ((15, 31), (32, 64)),
         ((31, 33), (62, 77)), ((25, 63), (50, 125)), ((45, 99), (90, 198)), ((63, 127), (128, 256)), ((3, 481), (9, 961)),
         ((341, 3), (686, 5)), ((3, 1023), (5, 2048)), ((3, 3125), (5, 6250)), ((1023, 5), (2048, 9)),
         ((1023, 1023), (2048, 2048)), ((3, 5, 7), (5, 9, 14)), ((15, 17, 33), (30, 34, 66)), ((33, 3, 41), (65, 7, 81))]


@pytest.mark.parametrize("N,M", GRIDS)
@pytest.mark.parametrize("tile,rows", [(0, 0), (1, 1), (4, 2), (16, 0)])
def test_operator_to_single_rounding(ghb, N, M, tile, rows):
    """Against the FP64 operator, within the rounding of a single-precision
    evaluation: log2|M| stages there and back, each within a few units of 2^-24
    of the norm (a prime stage p sums p terms, which log2 p stages cover)."""
    d = len(N)
    m = dict(d=d, N=list(N), a0=1.0, inclusions=[(0, (0.1, -0.2, 0.0), (0.5, 0.4, 0.3 if d == 3 else 0.0), 20.0)])
    kept = {n: ghb.tune_get(n) for n in set(M)}
    try:
        for n, cfg in kept.items():
            fits = tile * n * 8 * 17 // 16 <= 200 * 1024
            ghb.tune_set(n, **dict(cfg, tile32=tile if fits else 0, rows32=rows, ct_col=0, ct_row=0))
        ctx = ghb.Context.from_microstructure(m, M=tuple(M) + (0,) * (3 - d))
    finally:
        for n, cfg in kept.items():
            ghb.tune_set(n, **cfg)
    x = W.random_field(np.random.default_rng(sum(M)), d, list(N))
    xt = torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(x))).cuda()
    x32 = xt.to(torch.complex64)
    got, ref = ctx.matvec(x32).to(torch.complex128), ctx.matvec(x32.to(torch.complex128))
    tol = 4 * EPS * math.log2(max(math.prod(M), 2)) * math.sqrt(20.0)   # contrast 20: |A u| against |u|
    assert torch.linalg.norm(got - ref) <= tol * torch.linalg.norm(ref) + 1e-30


@pytest.mark.parametrize("count", [1, 6])
def test_batches_of_few_and_many_warps(ghb, count):
    """One instance of N = 255 stays below the 24 warps an SM that choose the kernels
    of 80 registers, six exceed them; either way the bounds are a single context's
    to the solves' tolerance, which the energies meet squared."""
    micros = [dict(d=2, N=[255, 255], a0=1.0, inclusions=[(1, (0.01 * i, -0.02 * i, 0.0), (0.31, 0.0, 0.0), 20.0 + i)])
              for i in range(count)]
    batch = ghb.Batch()
    for m in micros:
        batch.submit(m)
    batch.run()
    for m, r in zip(micros, sorted(batch.results(), key=lambda r: r["id"])):
        upper, lower, _, status = ghb.Context.from_microstructure(m, precision="mixed").bounds()
        assert status == 0
        for got, want in ((r["upper"], upper), (r["lower"], lower)):
            assert np.abs(np.asarray(got).reshape(2, 2) - want).max() <= 1e-10 * np.abs(want).max()
