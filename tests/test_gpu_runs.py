"""Work items that are runs of fluid cells, whose entries the step makes instead of reading
them: rows shorter than, equal to and longer than an item, odd and even, so that runs begin and
end at every place of a row, against the oracle; and a box large enough that the entries are
not asked for in advance."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _check(orc, g, storage, layout, n, tol):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    solid = orc.voxelize(g.shape, g.spheres)
    q = orc.wall_distances(solid, g.spheres)
    _, w, _ = orc.lattice()
    f0 = w[:, None, None, None] * (1.0 + 1e-3 * I.noise((19,) + g.shape, 8))
    f0[:, solid == 1] = 0.0
    kw = dict(tau=0.64, delta_rho=3e-4, magic_lambda=3 / 16, collision=capi.TRT, wall=capi.CLI)
    with capi.Context(spheres=g.spheres, shape=g.shape, storage=getattr(capi, storage),
                      layout=getattr(capi, "LAYOUT_" + layout), **kw) as ctx:
        ctx.set_populations(f0)
        ctx.step(n)
        f = ctx.get_populations()
    fref, _, _ = orc.run(solid, f0, n, q=q, **kw)
    fluid = solid == 0
    assert np.abs(f - fref)[:, fluid].max() / np.abs(fref)[:, fluid].max() <= tol


@pytest.mark.parametrize("nx", [31, 32, 33, 47, 64, 95])
@pytest.mark.parametrize("layout", ["AB", "AA"])
def test_runs_at_every_place_of_a_row(orc, nx, layout):
    _check(orc, I.Geometry(nx, 9, 10, np.array([[nx / 2 + 0.3, 4.6, 4.9, 3.1]])), "F64", layout, 9, 1e-12)


@pytest.mark.parametrize("layout", ["AB", "AA"])
def test_runs_of_a_large_box(orc, layout):
    _check(orc, I.Geometry(101, 110, 120, np.array([[40.3, 61.0, 55.2, 30.7]])), "F32", layout, 3, 1e-5)
