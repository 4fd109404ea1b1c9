"""Coefficient tables (csrc/fields.cu) at the edges of the kernel: inclusions held
64 at a time, every range of J_1 (8, 20, 40, 100), spheres near q = 0, boxes, odd
and small tables, one entry per mirror pair at n_0 = 0."""
import numpy as np
import pytest

import workloads as W
from oracle import coefficients as OC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


def disks(n, rng):
    side = int(np.ceil(np.sqrt(max(n, 1))))
    cells = [((i + 0.5) / side - 0.5, (j + 0.5) / side - 0.5) for i in range(side) for j in range(side)][:n]
    return [(1, (x, y, 0.0), (0.45 / side * rng.uniform(0.4, 1.0), 0.0, 0.0), float(rng.uniform(2, 50))) for x, y in cells]


@pytest.mark.parametrize("d,N,inc", [
    (2, (63, 45), 0), (2, (1, 1), 1), (2, (3, 127), 1), (2, (127, 3), 1), (2, (129, 129), 2), (2, (63, 45), 64), (2, (31, 45), 65),
    (2, (45, 33), 130), (2, (81, 27), "box"), (3, (5, 7, 33), "box"), (3, (17, 9, 21), "sphere"), (3, (3, 3, 1), "sphere")])
def test_table_edges(d, N, inc):
    """Per entry within the rounding of n.x_i (a few units of |n|_1 / 2, times 2 pi)
    and of the shape factors, each at most the inclusion's volume."""
    import paper_1412_2033_gb300 as ghb
    rng = np.random.default_rng(len(N) * 100 + sum(N))
    if inc == "box":
        incs = [(0, (-0.2, 0.1, 0.05), (0.37, 0.21, 0.6), 7.0), (0, (0.29, -0.23, 0.0), (0.11, 0.3, 0.25), 0.2)]
    elif inc == "sphere":
        incs = [(2, (-0.21, 0.13, 0.07), (0.2, 0.0, 0.0), 30.0), (2, (0.3, -0.3, 0.3), (1e-3, 0.0, 0.0), 5.0)]
    else:
        incs = disks(inc, rng)
    m = dict(d=d, N=list(N), a0=1.5, inclusions=incs)
    ctx = ghb.Context.from_microstructure(m)
    mat = OC.material_from_dict(m)
    k = np.abs(OC.freq_grid([2 * n - 1 for n in N])[..., N[-1] - 1:, :]).sum(-1)
    for kind, one in ((ghb.GHB_PRIMAL, mat), (ghb.GHB_DUAL, mat.inverse())):
        ref = OC.coeff_table(one, list(N))[..., N[-1] - 1:]
        got = ctx.table(kind).cpu().numpy()
        weight = sum(abs(i.value - one.a0) * f for i, f in zip(one.inclusions, one.volume_fractions())) if incs else 0.0
        assert (np.abs(got - ref) <= EPS * (2 * np.pi * k + 16) * weight + EPS * one.a0 * (k == 0)).all()


@pytest.mark.parametrize("d,N", [(2, 5), (2, 9), (2, 27), (3, 5), (3, 9)])
@pytest.mark.parametrize("h,center", [(0.37, 0.11), (0.21, 0.23), (0.5, -0.31)])
def test_laminate_loads_along_the_layers_need_no_iteration(d, N, h, center):
    """Their right-hand sides vanish: the projection keeps a component along an
    axis exactly, so no rounding residue is left to solve for."""
    import paper_1412_2033_gb300 as ghb
    for precision in ("fp64", "mixed"):
        ctx = ghb.Context.from_microstructure(W.laminate(N, d=d, h=h, value=8.0, a0=1.5, center=center), precision=precision)
        _, _, infos, status = ctx.bounds()
        assert status == 0
        assert all(infos[i]["iters"] == 0 for i in range(1, d + 1))   # upper: along the layers; lower: across them
