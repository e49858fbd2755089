"""The no-allocation moment sums of cells whose populations differ much in size are those of FP64
sums: small moving populations beside a large one at rest, zeros and subnormal values, and
fields whose largest population crosses a power of two from cell to cell, against exact sums.

Tolerance: a cell's FP64 sums and the additions after it (at most 18 in the cell, 1 a lane, 5 in
the warp, 8 in the block, 9 after it, 1 division) round at 2^-53 of the sum of the absolute
values that enter them, 48 * 2^-53 in all: of the moving ones for the momentum, which the
population at rest is no part of."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

E = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1],
              [1, 1, 0], [-1, -1, 0], [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1],
              [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1], [0, -1, 1]])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _field(kind, n):
    rng = np.random.default_rng(n)
    noise = rng.uniform(-1, 1, size=(19, n))
    f = W[:, None] * (1.0 + 1e-3 * noise)
    if kind.startswith("moving 2^"):
        f[1:] = noise[1:] * 2.0 ** int(kind[9:])
    elif kind == "zeros":
        f[1:] = np.where(rng.uniform(size=(18, n)) < 0.5, rng.choice([0.0, -0.0], size=(18, n)), f[1:])
    elif kind == "subnormal":
        f[1:] = 0.0
        f[1], f[8] = 1e-310, -3e-311
    elif kind == "crossing":
        f *= 1.5
    elif kind == "small beside":  # cells that are exact in integers beside cells that are not
        f[5, ::3] = 1e-7
    return f, 1.5 if kind == "crossing" else 1.0


@pytest.mark.parametrize("n", [1, 33, 20_000])
@pytest.mark.parametrize("kind", ["moving 2^-9", "moving 2^-20", "moving 2^-30", "moving 2^-60", "zeros", "subnormal",
                                  "crossing", "small beside"])
def test_sums_are_fp64_sums(n, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1508_02960_gb300 import capi
    f, rho0 = _field(kind, n)
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    fd = torch.from_numpy(f).cuda()
    capi.moment_sums_f64_noalloc(fd.data_ptr(), None, n, rho0, out.data_ptr(), torch.cuda.current_stream())
    got = out.cpu().numpy()
    ref = math.fsum(f.ravel().tolist() + [-rho0] * n)
    assert abs(got[0] - ref) <= 48 * 2.0 ** -53 * (np.abs(f).sum() + rho0 * n)
    for a in range(3):
        plus, minus = f[E[:, a] == 1], f[E[:, a] == -1]
        ref = math.fsum(plus.ravel().tolist() + (-minus).ravel().tolist()) / rho0
        size = (np.abs(plus).sum() + np.abs(minus).sum()) / rho0
        assert abs(got[1 + a] - ref) <= max(48 * 2.0 ** -53 * size, 5e-324), (a, got[1 + a], ref)
