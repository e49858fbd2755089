"""Flag fields so dense that a work item's cut links exceed a warp (up to 18 at each of its 32
cells, handled a warp at a time), against the oracle: both layouts, SBB and CLI, FP64 and FP32,
and the interpolated rules, whose fallbacks such a field exercises, in the A-B layout; with the
drag of the last step.  Tolerances per population as for the sphere cells: 1e-12 in FP64, 1e-5
in FP32, of the largest population."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi as C
    C.lib(build_if_missing=True)
    return C


def _field(shape, solid_share, seed):
    solid = (np.random.default_rng(seed).uniform(size=shape) < solid_share).astype(np.uint8)
    solid.reshape(-1)[::97] = 0  # some fluid at any share
    return solid


@pytest.mark.parametrize("shape,share", [((7, 9, 20), 0.55), ((5, 6, 33), 0.3), ((3, 4, 7), 0.8)])
@pytest.mark.parametrize("wall,layout", [("SBB", "AB"), ("SBB", "AA"), ("CLI", "AB"), ("CLI", "AA"), ("QIBB", "AB"),
                                         ("MR", "AB"), ("IEBB", "AB"), ("LIBB", "AB")])
@pytest.mark.parametrize("storage", ["F64", "F32"])
def test_dense_flag_fields_match_oracle(capi, orc, shape, share, wall, layout, storage):
    solid = _field(shape, share, 3)
    rng = np.random.default_rng(4)
    q = rng.uniform(0.05, 1.0, size=(19,) + shape)
    _, w, _ = orc.lattice()
    f0 = w[:, None, None, None] * (1.0 + 1e-3 * I.noise((19,) + shape, 6))
    f0[:, solid == 1] = 0.0
    kw = dict(tau=0.7, delta_rho=2e-4, magic_lambda=3 / 16, collision=capi.TRT, wall=getattr(capi, wall))
    n = 9
    with capi.Context(flags=solid, q=q, shape=shape, storage=getattr(capi, storage),
                      layout=getattr(capi, "LAYOUT_" + layout), **kw) as ctx:
        ctx.set_populations(f0)
        ctx.step(n)
        f = ctx.get_populations()
        o = ctx.observables()
    force = np.zeros(3)
    fref, sums, _ = orc.run(solid, f0, n, q=q, force=force, **kw)
    fluid = solid == 0
    err = np.abs(f - fref)[:, fluid].max() / np.abs(fref)[:, fluid].max()
    assert err <= (1e-12 if storage == "F64" else 1e-5), err
    # the force is a sum over the links of values of the size of the populations' deviations
    scale = 1e-3 * np.abs(w[1]) * max(1, int(fluid.sum())) * 18
    tol = 1e-12 if storage == "F64" else 1e-5
    assert np.abs(np.array([o["F_x"], o["F_y"], o["F_z"]]) - force).max() <= tol * scale
