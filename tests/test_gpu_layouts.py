"""Lines without (all of) their spare entries: forced column tiles that fill a CTA's
shared memory give the operator that the unforced ones give, to rounding."""
import math

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,tile64,tile32", [(768, 16, 16), (1536, 8, 16), (3072, 4, 8), (3128, 4, 8), (6144, 2, 4)])
def test_widest_forced_tiles(M, tile64, tile32):
    import numpy as np

    import paper_1412_2033_gb300 as ghb
    N = [min(M // 2 - 1 + (M // 2) % 2, (M + 1) // 2), 9]
    m = dict(d=2, N=N, a0=1.0, inclusions=[(0, (0.1, -0.2, 0.0), (0.5, 0.4, 0.0), 20.0)])
    x = torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(W.random_field(np.random.default_rng(M), 2, N)))).cuda()
    kept = ghb.tune_get(M)
    try:
        free = ghb.Context.from_microstructure(m, M=(M, 0, 0))
        ghb.tune_set(M, tile64=tile64, tile32=tile32, ct_col=0, ct_row=0)
        forced = ghb.Context.from_microstructure(m, M=(M, 0, 0))
    finally:
        ghb.tune_set(M, **kept)
    for dt, eps in ((torch.complex128, 2.0 ** -52), (torch.complex64, 2.0 ** -23)):
        a, b = free.matvec(x.to(dt)), forced.matvec(x.to(dt))
        tol = 4 * eps * math.log2(M * 18) * math.sqrt(20.0)   # two roundings of log2|M| stages, contrast 20
        assert torch.linalg.norm(a - b) <= tol * torch.linalg.norm(a)
