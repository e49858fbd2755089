"""A context that does not fit into the memory that is left (taken by another owner, so that the
allocation itself fails) is refused, and the next one, which fits, is created and steps."""
import pytest

from paper_1508_02960_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_next_context_after_a_refused_one():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    kw = dict(tau=0.7, delta_rho=1e-4, collision=capi.TRT, wall=capi.CLI)
    small = I.centred_sphere(24, 7.0)

    def steps():
        with capi.Context(spheres=small.spheres, shape=small.shape, storage=capi.F32, **kw) as ctx:
            ctx.init_equilibrium()
            ctx.step(20)
            return ctx.observables()["U_sup"]

    ref = steps()
    big = I.centred_sphere(320, 100.0)  # 10 GB of FP64 populations
    torch.cuda.empty_cache()
    taken = torch.empty(max(0, torch.cuda.mem_get_info()[0] - (2 << 30)), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(capi.LBMError) as e:
            capi.Context(spheres=big.spheres, shape=big.shape, storage=capi.F64, **kw)
        assert e.value.status == capi.ERR_NO_MEMORY
        assert steps() == ref
    finally:
        del taken
        torch.cuda.empty_cache()
