"""The autotuner's choice of the d = 3 last-axis kernels beside the d = 2 one."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_set_back_configuration_keeps_both_choices():
    """At M = 162 the size-specialised last-axis kernels are the faster ones for d = 3
    (47 us a pass at N = 81 against 66 and more), whatever d = 2 takes: the tuned
    operator is no slower than with ct_row = 0 forced, also after the configuration was
    read, changed and set back."""
    import paper_1412_2033_gb300 as ghb

    def application():
        ctx = ghb.Context(3, (81, 81, 81), 1.0, [(2, (0.1, -0.2, 0.0), (0.3,), 20.0)])
        assert ctx.M == [162, 162, 162]
        x = torch.ones(ctx.field_shape, dtype=torch.complex64, device="cuda")
        y = torch.empty_like(x)
        best = 1e30
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for _ in range(20):
                ctx.matvec(x, out=y)
            torch.cuda.synchronize()
            best = min(best, (time.perf_counter() - t) / 20)
        return best

    kept = ghb.tune_get(162)
    tuned = application()
    try:
        ghb.tune_set(162, **dict(kept, rows32=0, ct_row=0))
        general = application()
    finally:
        ghb.tune_set(162, **kept)
    assert ghb.tune_get(162) == kept
    back = application()
    assert tuned < 0.95 * general and back < 0.95 * general, (tuned, general, back)
