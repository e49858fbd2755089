"""FP64 fields to and from the host, in passes: several directions of a small box, a part of
one direction of a box of more than 2^20 cells (a third of that for the velocity)."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1),
              (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])


@pytest.fixture(scope="module")
def capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi as C
    C.lib(build_if_missing=True)
    return C


def _context(capi, shape, storage, layout, rho0=1.0):
    nx, ny, nz = shape
    r = 0.3 * min(shape)
    return capi.Context(spheres=np.array([[nx / 2, ny / 2, nz / 2, r]]), shape=shape[::-1], tau=0.7, delta_rho=1e-4, rho0=rho0,
                        collision=capi.TRT, wall=capi.CLI, storage=getattr(capi, storage),
                        layout=getattr(capi, "LAYOUT_" + layout))


def _velocity(f, rho0):
    m = np.tensordot(E.T.astype(float), f - W[:, None, None, None] * rho0, 1)
    return m / rho0


# 17 x 13 x 12: all directions in one pass; 64 x 32 x 33: 15 and 4; 96 x 80 x 72: one a pass,
# the velocity in two parts; 128 x 128 x 64: exactly 2^20; 104 x 101 x 100: two parts
@pytest.mark.parametrize("shape", [(17, 13, 12), (64, 32, 33), (96, 80, 72), (128, 128, 64), (104, 101, 100)])
@pytest.mark.parametrize("storage,layout,rho0", [("F64", "AB", 1.0), ("F32", "AA", 1.25)])
def test_round_trip(capi, shape, storage, layout, rho0):
    nz, ny, nx = shape[::-1]
    rng = np.random.default_rng(5)
    f = (W[:, None, None, None] * rho0 + 1e-3 * rng.uniform(-1, 1, (19, nz, ny, nx)))
    with _context(capi, shape, storage, layout, rho0) as ctx:
        solid = np.asarray(ctx.get_flags()).reshape(nz, ny, nx) != 0
        ctx.set_populations(f)
        out = np.asarray(ctx.get_populations()).reshape(f.shape)
        u = np.asarray(ctx.get_velocity()).reshape(3, nz, ny, nx)
        sums = np.asarray(ctx.moment_sums())
    # g rounds to 24 bits in FP32 (|g| <= 1e-3), f to 53 in either
    eps = 1e-3 * 2.0 ** -24 if storage == "F32" else 0.0
    assert np.abs(out - np.where(solid, 0.0, f)).max() <= eps + 2.0 ** -52
    assert np.abs(u[:, solid]).max() == 0.0
    want = np.where(solid, 0.0, _velocity(f, rho0))
    # at most 10 populations a component, each rounded, and their sum
    assert np.abs(u - want).max() <= 10 * eps + 2.0 ** -48
    n = (~solid).sum()
    got = np.concatenate([[sums[0]], sums[1:4]])
    exact = np.concatenate([[(f - W[:, None, None, None] * rho0)[:, ~solid].sum()], want[:, ~solid].sum(1)])
    assert np.abs(got - exact).max() <= n * (19 * eps + 2.0 ** -46)


@pytest.mark.parametrize("steps", [1, 2])
def test_in_place_layout_agrees(capi, steps):
    """After an odd step the AA state lies in the neighbours' slots."""
    shape = (96, 80, 72)
    out = []
    for layout in ("AB", "AA"):
        with _context(capi, shape, "F64", layout) as ctx:
            ctx.init_equilibrium()
            ctx.step(20 + steps)
            out.append([np.asarray(a) for a in (ctx.get_populations(), ctx.get_velocity(), ctx.moment_sums())])
    for a, b in zip(*out):  # same arithmetic in both layouts but for the order of sums
        assert np.abs(a - b).max() <= 1e-13 * max(1.0, np.abs(a).max())


@pytest.mark.parametrize("storage", ["F64", "F32"])
@pytest.mark.parametrize("k", [0, 1, 7])
def test_non_finite_populations_show(capi, storage, k):
    """An infinite population makes the cell's velocity infinite or NaN in every component,
    and no other cell's."""
    shape = (17, 13, 12)
    f = np.broadcast_to(W[:, None, None, None], (19, 12, 13, 17)).copy()
    f[k, 2, 3, 4] = np.inf
    with _context(capi, shape, storage, "AB") as ctx:
        ctx.set_populations(f)
        u = np.asarray(ctx.get_velocity()).reshape(3, 12, 13, 17)
        assert not np.isfinite(ctx.moment_sums()).any()
    bad = ~np.isfinite(u)
    assert bad[:, 2, 3, 4].all() and bad.sum() == 3
