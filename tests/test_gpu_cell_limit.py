"""GPU: the chain in the largest boxes that it takes, where the cells' counters
leave shared memory for fewer moves in flight than asked for (FP64: seven), move
by move against the oracle; one more cell per side is refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300._lib import GcmcError  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box, Mix  # noqa: E402

RC = 2.5
CELLS = {"fp64": 46, "fp32": 43}  # per side: 97,336 and 79,507 cells
TOL = {"fp64": 1e-12, "fp32": 1e-5}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("config", [0, 3])
def test_most_cells(precision, config):
    L, n = CELLS[precision] * RC + 0.1, 20_000
    pos = W.uniform_positions(n, L, 6)
    types = (np.arange(n) % 3 == 0).astype(np.int32)
    eps, sigma = W.lorentz_berthelot([1.0, 0.8], [1.0, 1.1])
    args = (0.3, 0.4, 0.3, 0.4, 1 / 1.2, [-4.0, -4.5])
    o = O.System(L, RC, eps, sigma)
    o.build(pos, types)
    o.set_energy(o.total_energy())
    b = Box(L, RC, eps, sigma, precision=precision)
    b.set_chain_config(config)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    assert b.geometry()["T"] == CELLS[precision]
    to, _ = o.run_moves(19, 0, 2000, *args, tol=TOL[precision])
    _, tg = b.run_moves(19, 0, 2000, Mix(*args), trace=True)
    for f in ("type", "species", "index", "accepted"):
        assert np.array_equal(tg[f], to[f]), f
    ok = np.isfinite(to["lnA"])
    assert np.all(np.abs(tg["dU"] - to["dU"])[ok] <= TOL[precision] * to["uabs"][ok] + 1e-300)
    for x, y in zip(o.state(), b.get_state()[:4]):
        assert np.array_equal(x, y)
    b.check_state()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_one_cell_more_is_refused(precision):
    L = (CELLS[precision] + 1) * RC + 0.1
    b = Box(L, RC, [[1.0]], [[1.0]], precision=precision)
    b.build_cells(torch.as_tensor(W.uniform_positions(100, L, 6)), torch.zeros(100, dtype=torch.int32))
    with pytest.raises(GcmcError, match="too many cells"):
        b.run_moves(19, 0, 10, Mix(0.3, 0.4, 0.3, 0.4, 1.0, [-4.0]))
