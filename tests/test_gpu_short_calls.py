"""Calls of few steps of a batch of several groups step all instances in one launch a step, longer
ones group by group: the launches of either, and, with both kinds in turn and odd and even counts,
every instance's state and observables bit for bit as alone; batches beyond the tile map's
instances, too."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CALLS = (1, 6, 2, 3, 60, 1, 5, 7, 4)


@pytest.mark.parametrize("layout", ["AB", "AA"])
@pytest.mark.parametrize("geoms", [[(80, 12.0), (24, 7.0), (81, 11.0), (17, 5.0)], [(40, 9.0)] * 70], ids=["4", "70"])
def test_short_and_long_calls(layout, geoms):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    geoms = [I.centred_sphere(L, r + 0.01 * i) for i, (L, r) in enumerate(geoms)]
    keep = [capi.make_desc(spheres=g.spheres, shape=g.shape, tau=0.6 + 0.001 * i, delta_rho=1e-4 * (1 + i),
                           collision=capi.TRT, wall=capi.CLI, storage=capi.F32,
                           layout=getattr(capi, "LAYOUT_" + layout)) for i, g in enumerate(geoms)]
    b = capi.Batch([d for d, _ in keep])
    b.init_equilibrium()
    for n in CALLS:
        before = b.info()["kernel_launches"]
        b.step(n)
        made = b.info()["kernel_launches"] - before
        # a step of all instances and the final sums; of several groups each takes its steps
        assert made == n + 1 if n <= 5 else made > n + 1 and (made - 1) % n == 0, (n, made)
    got = [(b.get_populations(i), b.observables(i)) for i in range(len(keep))]
    b.close()
    for i in (0, 1, 2, 3, len(keep) - 1):
        with capi.Context(desc=keep[i][0]) as ctx:
            ctx.init_equilibrium()
            for n in CALLS:
                ctx.step(n)
            assert np.array_equal(ctx.get_populations(), got[i][0])
            o = ctx.observables()
        for k in ("U_sup", "mass", "F_x", "F_y", "F_z", "K", "steps", "n_fluid"):
            assert o[k] == got[i][1][k], k


def test_fp64_instances_step_together():
    """FP64 instances, whatever their size, share every launch."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    geoms = [I.centred_sphere(80, 12.0), I.centred_sphere(24, 7.0), I.centred_sphere(76, 11.0)]
    keep = [capi.make_desc(spheres=g.spheres, shape=g.shape, tau=0.6 + 0.01 * i, delta_rho=1e-4, collision=capi.TRT,
                           wall=capi.CLI, storage=capi.F64) for i, g in enumerate(geoms)]
    b = capi.Batch([d for d, _ in keep])
    b.init_equilibrium()
    for n in (60, 7):
        before = b.info()["kernel_launches"]
        b.step(n)
        assert b.info()["kernel_launches"] - before == n + 1
    got = [b.get_populations(i) for i in range(3)]
    b.close()
    for (d, _), f in zip(keep, got):
        with capi.Context(desc=d) as ctx:
            ctx.init_equilibrium()
            for n in (60, 7):
                ctx.step(n)
            assert np.array_equal(ctx.get_populations(), f)
