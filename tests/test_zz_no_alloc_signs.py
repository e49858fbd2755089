"""The no-allocation moment sums do not depend on the direction of the flow: a weak flow along -x
and the same flow along +x have equal and opposite sums, each as accurate as the other."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

E = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1],
              [1, 1, 0], [-1, -1, 0], [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1],
              [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1], [0, -1, 1]])
OPP = [0] + [k + 1 if k % 2 else k - 1 for k in range(1, 19)]
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.fixture(scope="module")
def capi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi as C
    C.lib(build_if_missing=True)
    return C


def _sums(capi, f, rho0=1.0):
    import torch
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    fd = torch.from_numpy(np.ascontiguousarray(f)).cuda()
    capi.moment_sums_f64_noalloc(fd.data_ptr(), None, f.shape[1], rho0, out.data_ptr(), torch.cuda.current_stream())
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [1, 300, 20_000])
@pytest.mark.parametrize("u", [1e-12, 1e-6])
def test_weak_flow_against_an_axis(capi, n, u):
    """Every block's sum has the flow's sign, so the additions after the blocks' exact sums (at
    most 64 in a row, and the two roundings of each block's value) are good to 66 * 2^-53."""
    rng = np.random.default_rng(n)
    rho = 1.0 - 1e-9 * rng.uniform(0.5, 1.0, size=n)     # a density sum below zero, too
    f = W[:, None] * rho * (1.0 + 3.0 * u * E[:, :1])
    plus, minus = _sums(capi, f), _sums(capi, f[OPP])
    assert plus[0] == minus[0] and np.array_equal(plus[1:], -minus[1:])
    ref = math.fsum(f[E[:, 0] == 1].ravel().tolist() + (-f[E[:, 0] == -1]).ravel().tolist())
    drho = math.fsum(f.ravel().tolist() + [-1.0] * n)
    assert ref > 0.0 and drho < 0.0
    assert abs(plus[1] - ref) <= 66 * 2.0 ** -53 * ref
    assert abs(plus[0] - drho) <= 66 * 2.0 ** -53 * -drho
