"""GPU: the microcell chain against the oracle for cubes that the usual edge and
step do not give: displacements of several cells (two cubes), edges below and
above a third of the cutoff, a box that one cube spans.  Same decisions, dU
within tol * uabs as for the usual shapes (1e-12 FP64, 1e-5 FP32: plain FP32
terms), same lists afterwards."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box, Mix  # noqa: E402

TOL = {"fp64": 1e-12, "fp32": 1e-5}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,L,rc,S,edge,step", [(900, 12.0, 2.5, 1, 1.0, 4.5), (900, 12.0, 2.5, 2, 0.55, 0.3),
                                                (700, 11.2, 2.5, 2, 2.0, 0.4), (150, 7.5, 2.5, 1, 1.9, 3.0)])
def test_cube_shapes(precision, n, L, rc, S, edge, step):
    rng = np.random.default_rng(n)
    side = int(np.ceil(n ** (1 / 3)))
    site = rng.permutation(side ** 3)[:n]
    ijk = np.stack([site % side, site // side % side, site // side ** 2], 1)
    pos = ((ijk + 0.5 + rng.uniform(-0.1, 0.1, (n, 3))) * (L / side)) % L
    types = (np.arange(n) % 5 == 0).astype(np.int32) * (S - 1)
    eps, sigma = W.lorentz_berthelot([1.0, 0.8][:S], [1.0, 1.1][:S])
    o = O.System(L, rc, eps, sigma)
    o.build(pos, types)
    o.set_energy(o.total_energy())
    b = Box(L, rc, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    o.micro_build(edge)
    b.build_microcells(edge)
    args = (0.5, 0.25, 0.25, step, 1 / 1.3, [-2.5] * S)
    to, so = o.run_moves(11, 0, 6000, *args, tol=TOL[precision])
    sg, tg = b.run_moves_micro(11, 0, 6000, Mix(*args), trace=True)
    for k in ("type", "species", "index", "accepted"):
        assert np.array_equal(tg[k], to[k]), k
    ok = np.isfinite(to["lnA"])
    assert np.all(np.abs(tg["dU"] - to["dU"])[ok] <= TOL[precision] * to["uabs"][ok] + 1e-300)
    assert sg["accepted"] == list(so.accepted) and sum(sg["accepted"]) > 0
    for x, y in zip(o.state(), b.get_state()[:4]):
        assert np.array_equal(x, y)
    M_o, cnt_o, refs_o, _ = o.micro_state()
    M, cap, cnt, slots = b.microcells()
    assert M == M_o and np.array_equal(cnt.astype(np.int64), cnt_o)
    k = np.arange(cap)[:, None] < cnt[None, :].astype(np.int64)
    assert np.array_equal(slots[:, :, 3].T[k.T], refs_o)
