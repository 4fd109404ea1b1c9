"""The FP64 operator on the fixed-point transforms (csrc/fft_fx.cuh) where it can
go wrong: every pass shape and padding, prime stages, exponents at the ends of
the double range, lines of very different size, zeros, infinities and NaN."""
import math

import numpy as np
import pytest

import workloads as W
from oracle import coefficients as OC
from oracle import galerkin as OG

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def ghb():
    import paper_1412_2033_gb300 as g
    g.load_library()
    return g


def apply(ghb, ctx, x, kind=0):
    xt = torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(x))).cuda()
    return ctx.matvec(xt, kind=kind).cpu().numpy()


# double grids: groups of 2 .. 10 entries, padded (8) and not, primes 7 .. 31, one pass, many passes
GRIDS = [((1, 3), (1, 5)), ((3, 5), (8, 9)), ((9, 15), (17, 29)), ((13, 15), (25, 31)), ((16 - 1, 31), (32, 64)),
         ((31, 33), (62, 77)), ((25, 63), (50, 125)), ((41, 81), (81, 162)), ((45, 99), (90, 198)), ((63, 127), (128, 256)),
         ((3, 511), (6, 1024)), ((5, 481), (9, 961)), ((3, 1023), (5, 2048)), ((3, 2187), (5, 4374)), ((3, 3125), (5, 6250))]


@pytest.mark.parametrize("N,M", GRIDS)
@pytest.mark.parametrize("kind", [0, 1])
def test_operator_to_rounding(ghb, N, M, kind):
    """Within the rounding of a double-precision evaluation: both sides transform
    log2|M| stages there and back, each within a few units of 2^-53 of the norm."""
    m = dict(d=2, N=list(N), a0=1.0, inclusions=[(0, (0.1, -0.2, 0.0), (0.5, 0.4, 0.0), 20.0)])
    x = W.random_field(np.random.default_rng(sum(M)), 2, list(N))
    ref = ghb.half_from_full(OG.Operator(OC.material_from_dict(m), list(N), (OG.PRIMAL, OG.DUAL)[kind], M=list(M)).apply(x))
    ctx = ghb.Context.from_microstructure(m, M=(*M, 0))
    got = apply(ghb, ctx, x, kind)
    tol = 4 * EPS * math.log2(max(M[0] * M[1], 2)) * np.sqrt(20.0)   # contrast 20: |A u| against |u|
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("shift", [-900, -300, 300, 800])
def test_scaling_by_powers_of_two_is_exact(ghb, shift):
    m = W.random_disk_instance(3, N=31)
    ctx = ghb.Context.from_microstructure(m)
    x = W.random_field(np.random.default_rng(0), 2, m["N"])
    a, b = apply(ghb, ctx, x), apply(ghb, ctx, x * 2.0 ** shift)
    assert np.array_equal(a * 2.0 ** shift, b)


def test_columns_of_different_size_keep_their_own_precision(ghb):
    """Every line has its own exponent: a constant coefficient multiplies each
    frequency by a0, whatever the size of the others (2 on a plane k_1 = const,
    1e-200 elsewhere in the last axis' direction)."""
    N = [45, 33]
    ctx = ghb.Context(2, N, 3.0, [])
    x = W.random_field(np.random.default_rng(1), 2, N)
    s = np.ones(33)
    s[16] = 1e200
    y = ctx.matvec(torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(x * s))).cuda(), project=False).cpu().numpy()
    ref = 3.0 * ghb.half_from_full(x * s)
    assert np.abs(y - ref).max() <= 1e-14 * np.abs(ref).max()


def test_zero_and_non_finite_fields(ghb):
    m = W.random_disk_instance(5, N=33)
    ctx = ghb.Context.from_microstructure(m)
    x = W.random_field(np.random.default_rng(2), 2, m["N"])
    assert not apply(ghb, ctx, np.zeros_like(x)).any()
    for bad in (np.nan, np.inf, -np.inf):
        z = x.copy()
        z[0, 3, 20] = bad
        y = apply(ghb, ctx, z)
        y[:, 16, 0] = np.nan                     # k = 0 is projected to zero
        assert not np.isfinite(y).any()
