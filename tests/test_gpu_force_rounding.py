"""GPU: the forces of isolated pairs whose r U'(r) is exact, so that nothing but
the division by r^2 and the product with the separation is rounded.

eps = 1/4, sigma = r = m / 2048 (m < 4096) and a grid spacing that is a power of
two: (sigma / r)^2 = 1, 4 eps = 1, r U'(r) = -6, and r^2 and the separation are
floats.  dE/dx = fl(fl(-6 / r^2) r) times powers of two, two roundings: within
(1 + 2^-24)^2 - 1 of -6 / r.  A reciprocal of r^2 that is rounded first would add
a third; the 36 values of m are those where that misses the bound or comes
closest to missing it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1408_3764_gb300.gcmc import Box  # noqa: E402

BOUND = (1 + 2.0 ** -24) ** 2 - 1


def _hard_values():
    m = np.arange(2048, 4096)
    f = m.astype(np.float32)
    got = ((np.float32(1) / (f * f)) * np.float32(-6)) * f
    return m[np.argsort(-np.abs(got.astype(np.float64) * m / -6.0 - 1.0), kind="stable")[:36]]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_two_roundings(precision):
    S, L = 8, 64.0
    pairs = [(a, b) for a in range(S) for b in range(a, S)]
    r = _hard_values() / 2048.0
    sigma = np.empty((S, S))
    pos = np.empty((2 * len(pairs), 3))
    types = np.empty(2 * len(pairs), np.int32)
    half = L / 2.0 ** 33  # centres of grid points
    for k, (a, b) in enumerate(pairs):
        sigma[a, b] = sigma[b, a] = r[k]
        pos[2 * k] = pos[2 * k + 1] = (10.0 * (k % 6) + 3.0 + half, 10.0 * (k // 6) + 3.0 + half, 7.0 + half)
        pos[2 * k + 1, 0] += r[k]
        types[2 * k], types[2 * k + 1] = a, b
    box = Box(L, 2.5, np.full((S, S), 0.25), sigma, precision=precision)
    box.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    d = box.energy_grad(input_order=True)["dpos"].cpu().numpy().astype(np.float64)
    assert np.all(d[:, 1:] == 0.0)
    # the left particle gains energy as it moves towards the right one
    for got, sign in ((d[0::2, 0], 1.0), (d[1::2, 0], -1.0)):
        err = np.abs(got / (sign * 6.0 / r) - 1.0)
        assert err.max() <= BOUND, err.max() / 2.0 ** -24
