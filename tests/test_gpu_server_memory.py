"""The request loop when device memory runs out while a point joins points that are resident (every
allocation from the joining point's first on failed in turn, from the host): the batch they
share is usable again once memory is there, and serves the next point as a context of its own
steps it, bit for bit."""
import time

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


def _point(capi, L, r):
    g = I.centred_sphere(L, r)
    return capi.make_desc(spheres=g.spheres, shape=g.shape, tau=0.7, delta_rho=1e-4, collision=capi.TRT,
                          wall=capi.CLI, storage=capi.F32)


def _wait(poll, limit=60.0):
    t0 = time.time()
    while True:
        got = poll()
        if got:
            return got
        assert time.time() - t0 < limit
        time.sleep(0.005)


def _join_without_memory(capi, srv, n):
    """A point joins a resident one while every allocation but the first n fails; returns the
    resident point's id and whether an allocation failed."""
    d1, _k1 = _point(capi, 16, 5.0)
    r1 = srv.submit(d1, 1e-30, 10 ** 8)
    _wait(lambda: srv.stats()["fluid_updates"] > 0)
    d2, _k2 = _point(capi, 20, 6.0)
    capi.debug_fail_alloc_after(n)
    try:
        r2 = srv.submit(d2, 1e-30, 10 ** 8)
        t0 = time.time()
        while srv.poll(r2) is None and time.time() - t0 < 1.0:
            time.sleep(0.005)
        time.sleep(0.02)                  # (some chunks)
    finally:
        capi.debug_fail_alloc_after(-1)
    failed = srv.poll(r2) is not None
    if not failed:
        srv.cancel(r2)
        _wait(lambda: srv.poll(r2))
    return r1, failed


def test_batch_is_usable_after_a_failed_join(capi):
    d3, _k3 = _point(capi, 24, 7.0)
    with capi.Context(desc=d3) as ctx:
        ctx.init_equilibrium()
        ctx.step(400)
        alone = ctx.observables()["U_sup"]
    for n in range(100):
        srv = capi.Server(hbm_budget_bytes=1 << 30, check_interval=50, max_resident=4)
        try:
            r1, failed = _join_without_memory(capi, srv, n)
            if srv.poll(r1) is None:
                srv.cancel(r1)
                _wait(lambda: srv.poll(r1))
            r3 = srv.submit(d3, 1e-30, 400)
            st, obs, _ = _wait(lambda: srv.poll(r3))
            assert st == capi.ERR_NOT_CONVERGED and obs["steps"] == 400 and obs["U_sup"] == alone, n
        finally:
            srv.close()
        if not failed:
            break                          # n allocations suffice: every failure was met
    assert 10 < n < 99


def test_resident_point_is_not_judged_by_a_failed_step(capi):
    """A resident point whose steps fail for want of memory is reported so (or steps on), never as
    converged on the numbers of the step before."""
    met = 0
    for n in range(100):
        srv = capi.Server(hbm_budget_bytes=1 << 30, check_interval=50, max_resident=4)
        try:
            r1, failed = _join_without_memory(capi, srv, n)
            got = srv.poll(r1)
            assert got is None or got[0] == capi.ERR_NO_MEMORY, (n, got and got[0])
            met += got is not None
        finally:
            srv.close()
        if not failed:
            break
    assert met > 0
