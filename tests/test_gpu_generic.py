"""Stages of every prime radix 7 .. 31 (csrc/fft_rt.cuh, fft_fx.cuh): as the only pass,
the first, the last and both, FP32 against FP64 and FP64 against the oracle."""
import math

import numpy as np
import pytest

import workloads as W
from oracle import coefficients as OC
from oracle import galerkin as OG

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [7, 11, 13, 17, 19, 23, 29, 31])
@pytest.mark.parametrize("M", [(1, 2), (2, 1), (9, 1), (0, 4)])   # times p; 0: p^2
def test_prime_stages(p, M):
    import paper_1412_2033_gb300 as ghb
    M = [p * m if m else p * p for m in M]
    N = [(m + 1) // 2 - 1 + (m + 1) // 2 % 2 for m in M]
    m = dict(d=2, N=N, a0=1.0, inclusions=[(0, (0.1, -0.2, 0.0), (0.5, 0.4, 0.0), 20.0)])
    ctx = ghb.Context.from_microstructure(m, M=(*M, 0))
    x = W.random_field(np.random.default_rng(sum(M)), 2, N)
    ref = ghb.half_from_full(OG.Operator(OC.material_from_dict(m), N, OG.PRIMAL, M=M).apply(x))
    x64 = torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(x))).cuda()
    got = ctx.matvec(x64)
    # log2|M| stages there and back, each within a few units in the last place; contrast 20
    tol = 4 * math.log2(M[0] * M[1]) * math.sqrt(20.0)
    assert np.linalg.norm(got.cpu().numpy() - ref) <= tol * 2.0 ** -52 * np.linalg.norm(ref)
    x32 = x64.to(torch.complex64)
    a, b = ctx.matvec(x32).to(torch.complex128), ctx.matvec(x32.to(torch.complex128))
    assert torch.linalg.norm(a - b) <= tol * 2.0 ** -23 * torch.linalg.norm(b)
