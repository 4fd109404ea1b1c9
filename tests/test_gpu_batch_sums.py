"""The inner products of batched solves: independent of the batch's other requests,
and FP32 ones no coarser than one entry's sum however many entries a thread takes."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("others", [12, 40])
def test_alone_equals_in_a_large_mix(others):
    """The sums of a solve are split by its own size, so the bounds and the iteration
    counts of a request are the same bits alone and beside any number of others."""
    import paper_1412_2033_gb300 as ghb
    target = W.random_disk_instance(W.BASE_SEED + 99, N=255)

    def bounds(extra):
        b = ghb.Batch()
        rid = b.submit(target)
        for i in range(extra):
            b.submit(W.random_disk_instance(W.BASE_SEED + 400 + i, N=201 + 2 * (i % 28)))
        b.run()
        r = {r["id"]: r for r in b.results()}[rid]
        b.close()
        return r

    alone, mixed = bounds(0), bounds(others)
    assert alone["status"] == mixed["status"] == 0
    assert np.array_equal(alone["upper"], mixed["upper"]) and np.array_equal(alone["lower"], mixed["lower"])
    assert [i["iters"] for i in alone["infos"]] == [i["iters"] for i in mixed["infos"]]
