"""Batches whose instances step in several groups (one large enough to fill the GPU alone, the
others together): every instance reaches the state and the observables it reaches alone, bit
for bit, over calls that tune the block shapes and calls that do not, with an even and an odd
number of steps."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["AB", "AA"])
@pytest.mark.parametrize("storage", ["F32", "F16DEV"])
def test_groups_step_as_alone(layout, storage):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    geoms = [I.centred_sphere(24, 7.3), I.centred_sphere(80, 12.0), I.Geometry(31, 18, 20, np.array([[5.5, 9.0, 8.2, 6.7]])),
             I.centred_sphere(16, 5.1)]
    keep = [capi.make_desc(spheres=g.spheres, shape=g.shape, tau=0.6 + 0.02 * i, delta_rho=1e-4 * (1 + i),
                           collision=capi.TRT, wall=capi.CLI, storage=getattr(capi, storage),
                           layout=getattr(capi, "LAYOUT_" + layout)) for i, g in enumerate(geoms)]
    b = capi.Batch([d for d, _ in keep])
    b.init_equilibrium()
    for n in (60, 2, 7):
        b.step(n)
    got = [(b.get_populations(i), b.observables(i)) for i in range(len(keep))]
    b.close()
    for (d, _), (f, o) in zip(keep, got):
        with capi.Context(desc=d) as ctx:
            ctx.init_equilibrium()
            for n in (60, 2, 7):
                ctx.step(n)
            assert np.array_equal(ctx.get_populations(), f)
            oa = ctx.observables()
        assert oa["status"] == o["status"]
        for k in ("U_sup", "mass", "F_x", "F_y", "F_z", "K", "steps", "n_fluid"):
            assert oa[k] == o[k], k
