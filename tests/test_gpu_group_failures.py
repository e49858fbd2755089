"""A call of a batch during which the steps of a group can no longer be recorded (an injected
failure on the host) is refused without a step taken, when nothing is queued yet, or goes through;
either way every instance is at the state that it reaches alone in the steps that it reports, bit
for bit, and the next call goes on from there."""
import numpy as np
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def capi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi as C
    C.lib(build_if_missing=True)
    yield C
    C.debug_fail_alloc_after(-1)


def _descs(capi, layout, k):
    """Three groups: two cells that fill the GPU alone, and two small ones.  k varies the radii, so
    that the shapes of no group are known."""
    geoms = [I.centred_sphere(24, 7.0 + 0.4 * k), I.centred_sphere(80, 12.0 + 0.3 * k), I.centred_sphere(84, 9.0 + 0.3 * k),
             I.centred_sphere(18, 5.0 + 0.2 * k)]
    return [capi.make_desc(spheres=g.spheres, shape=g.shape, tau=0.6 + 0.02 * i, delta_rho=1e-4 * (1 + i),
                           collision=capi.TRT, wall=capi.CLI, storage=capi.F32,
                           layout=getattr(capi, "LAYOUT_" + layout)) for i, g in enumerate(geoms)]


def _step_without_memory(capi, b, n, k):
    """True if a step call of which the k-th recording fails is refused."""
    capi.debug_fail_alloc_after(k)
    try:
        b.step(n)
        return False
    except capi.LBMError as e:
        assert e.status == capi.ERR_NO_MEMORY
        return True
    finally:
        capi.debug_fail_alloc_after(-1)


def _same_as_alone(capi, keep, b):
    at = []
    for i, (d, _) in enumerate(keep):
        f, o = b.get_populations(i), b.observables(i)
        with capi.Context(desc=d) as ctx:
            ctx.init_equilibrium()
            ctx.step(o["steps"])
            assert np.array_equal(ctx.get_populations(), f), i
            assert ctx.observables()["U_sup"] == pytest.approx(o["U_sup"], rel=1e-6)
        at.append(o["steps"])
    return at


@pytest.mark.parametrize("layout", ["AB", "AA"])
def test_recording_fails_at_each_group(capi, layout):
    keep = _descs(capi, layout, 0)
    b = capi.Batch([d for d, _ in keep])
    b.init_equilibrium()
    b.step(8)
    done = 8
    for k in range(4):                          # three groups record the steps of a new count
        n = 9 + k
        refused = _step_without_memory(capi, b, n, k)
        assert refused == (k == 0)
        done += 0 if refused else n
        assert _same_as_alone(capi, keep, b) == [done] * 4
        b.step(n)
        done += n
        assert _same_as_alone(capi, keep, b) == [done] * 4
    b.close()


@pytest.mark.parametrize("layout", ["AB", "AA"])
def test_recording_fails_while_the_shapes_are_timed(capi, layout):
    for k in range(13):                         # three shapes and the steps, of three groups
        keep = _descs(capi, layout, k + 1)
        b = capi.Batch([d for d, _ in keep])
        b.init_equilibrium()
        refused = _step_without_memory(capi, b, 61, k)
        assert refused == (k < 3)
        assert _same_as_alone(capi, keep, b) == [0 if refused else 61] * 4
        b.step(61)
        assert _same_as_alone(capi, keep, b) == [61 if refused else 122] * 4
        b.close()
