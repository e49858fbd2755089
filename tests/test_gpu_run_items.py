"""Steps that make the entries of run items instead of reading them: those of a state (of the
instances stepping together) above 64 MiB, at row lengths where runs begin and end at every
place of a row and where a run is a whole row of 32 cells, whose first and last cell both lie on
an x face.

Against the oracle, and bit for bit against steps that read the entries: the FP64 state of
about 290,000 fluid cells is above the limit in the A-B layout and below it in place, where the
two layouts agree; in a batch, in-place instances that step together are above it."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIMIT = 64 << 20
KW = dict(tau=0.64, delta_rho=3e-4, magic_lambda=3 / 16)


@pytest.fixture(scope="module")
def capi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi as C
    C.lib(build_if_missing=True)
    return C


def _geometry(nx, cells, at=0.5):
    """About `cells` cells in rows of nx, with a sphere that leaves most rows whole."""
    ny = round((cells / nx) ** 0.5)
    nz = round(cells / nx / ny)
    return I.Geometry(nx, ny, nz, np.array([[at * nx + 0.3, ny / 3 + 0.2, nz / 2 + 0.1, 9.4]]))


def _start(orc, g, seed):
    solid = orc.voxelize(g.shape, g.spheres)
    _, w, _ = orc.lattice()
    f = w[:, None, None, None] * (1.0 + 1e-3 * I.noise((19,) + g.shape, seed))
    f[:, solid == 1] = 0.0
    return solid, f


def _run(capi, g, f0, layout, storage, n):
    with capi.Context(spheres=g.spheres, shape=g.shape, storage=getattr(capi, storage), collision=capi.TRT,
                      wall=capi.CLI, layout=getattr(capi, "LAYOUT_" + layout), **KW) as ctx:
        ctx.set_populations(f0)
        ctx.step(n)
        return ctx.get_populations(), ctx.info()["n_fluid"]


@pytest.mark.parametrize("storage,layout,cells,n", [("F64", "AB", 32 * 96 * 96, 5), ("F64", "AB", 32 * 96 * 96, 6),
                                                    ("F32", "AA", 32 * 170 * 170, 5), ("F32", "AA", 32 * 170 * 170, 6)])
def test_rows_of_one_run_match_oracle(capi, orc, storage, layout, cells, n):
    g = _geometry(32, cells)
    solid, f0 = _start(orc, g, 8)
    f, nf = _run(capi, g, f0, layout, storage, n)
    assert nf * 19 * (8 if storage == "F64" else 4) * (2 if layout == "AB" else 1) > LIMIT
    q = orc.wall_distances(solid, g.spheres)
    fref, _, _ = orc.run(solid, f0, n, q=q, collision=capi.TRT, wall=capi.CLI, **KW)
    fluid = solid == 0
    assert np.abs(f - fref)[:, fluid].max() / np.abs(fref)[:, fluid].max() <= (1e-12 if storage == "F64" else 1e-5)


@pytest.mark.parametrize("nx", [32, 33, 47, 64, 95])
@pytest.mark.parametrize("n", [5, 6])
def test_made_entries_step_as_read_ones(capi, orc, nx, n):
    g = _geometry(nx, 295_000)
    _, f0 = _start(orc, g, 3 + n)
    made, nf = _run(capi, g, f0, "AB", "F64", n)
    read, _ = _run(capi, g, f0, "AA", "F64", n)
    assert nf * 19 * 8 <= LIMIT < nf * 19 * 16
    assert np.array_equal(made, read)


@pytest.mark.parametrize("nx", [32, 47])
def test_made_entries_of_a_group(capi, orc, nx):
    geoms = [_geometry(nx, 290_000, at) for at in (0.3, 0.5, 0.7)]
    states = [_start(orc, g, 20 + i)[1] for i, g in enumerate(geoms)]
    keep = [capi.make_desc(spheres=g.spheres, shape=g.shape, collision=capi.TRT, wall=capi.CLI, storage=capi.F64,
                           layout=capi.LAYOUT_AA, **KW) for g in geoms]
    b = capi.Batch([d for d, _ in keep])
    for i, f in enumerate(states):
        b.set_populations(i, f)
    nf = b.info()["n_fluid"]
    assert nf / 3 * 19 * 8 <= LIMIT < nf / 3 * 2 * 19 * 8
    for n in (5, 2):
        b.step(n)
    got = [b.get_populations(i) for i in range(3)]
    b.close()
    for (d, _), f0, f in zip(keep, states, got):
        with capi.Context(desc=d) as ctx:
            ctx.set_populations(f0)
            for n in (5, 2):
                ctx.step(n)
            assert np.array_equal(ctx.get_populations(), f)
