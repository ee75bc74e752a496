"""GPU: the cell list against the oracle where the build changes its kernels:
the cell counts scanned by one block or by three kernels (16,384 cells lie
between T = 25 and 26), one pass of the former or several, one species (ranked
by input index) or more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box  # noqa: E402


@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("T,n", [(3, 5), (15, 4000), (16, 4001), (17, 1), (25, 9000), (26, 9001)])
def test_build(T, n, S):
    rc = 2.5
    L = (T + 0.3) * rc
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=rc, n_species=S, seed=T)
    o = O.System(L, rc, eps, sigma)
    cl = o.build(pos, types)
    b = Box(L, rc, eps, sigma)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    assert b.geometry()["T"] == T
    cs, cc, order = b.cell_list()
    assert np.array_equal(cc.cpu().numpy(), cl.cell_count)
    assert np.array_equal(cs.cpu().numpy(), cl.cell_start)
    assert np.array_equal(order.cpu().numpy(), cl.order)
    for x, y in zip(o.state(), b.get_state()[:4]):
        assert np.array_equal(x, y)
