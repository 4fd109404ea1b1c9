"""Every line of the FP64 (fixed-point) transforms has its own exponent."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [(15, 31), (45, 33), (121, 81)])
@pytest.mark.parametrize("a,b", [(150, -150), (-200, 100), (0, -60)])
def test_fields_of_different_size_in_one_gram_pass(N, a, b):
    """d = 2 Gram matrices transform both fields in one launch, their lines side by side.
    Scaling the fields by powers of two moves the lines' exponents and nothing else, so
    the entries scale exactly; with one exponent for both the smaller field would be
    lost (60 binary places below the larger one)."""
    import paper_1412_2033_gb300 as ghb
    m = dict(d=2, N=list(N), a0=1.0, inclusions=[(0, (0.1, -0.2, 0.0), (0.5, 0.4, 0.0), 20.0)])
    ctx = ghb.Context.from_microstructure(m)
    rng = np.random.default_rng(sum(N))
    u, v = (torch.from_numpy(np.ascontiguousarray(ghb.half_from_full(W.random_field(rng, 2, list(N))))).cuda() for _ in range(2))
    plain = ctx.gram(0, [u, v])
    scaled = ctx.gram(0, [u * 2.0 ** a, v * 2.0 ** b])
    assert np.array_equal(scaled, plain * np.array([[2.0 ** (2 * a), 2.0 ** (a + b)], [2.0 ** (a + b), 2.0 ** (2 * b)]]))
