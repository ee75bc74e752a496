"""The chain kernel where its speculative moves get in each other's way, against
the oracle move by move: boxes of three cells per side in which every accepted
move voids the moves in flight, crowded cells (more than 32 entries), deletions
that refill from a particle just inserted, moves in flight beyond the launch's
last move, and several species."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_1408_3764_gb300 import workloads as W
from paper_1408_3764_gb300.gcmc import Box, Mix

pytestmark = pytest.mark.gpu

# (n, L, rc, species, eps, (p_disp, p_ins, p_del), max_disp, ln z, moves)
CASES = {
    "ideal_crowded": (900, 6.0, 2.0, 1, 0.0, (0.2, 0.4, 0.4), 0.5, math.log(4.2), 3000),
    "ideal_sparse": (12, 5.01, 2.5, 1, 0.0, (0.2, 0.4, 0.4), 0.5, math.log(0.1), 3000),
    "empties": (4, 6.0, 2.0, 2, 0.0, (0.1, 0.2, 0.7), 0.5, math.log(0.02), 2000),
    "mixture": (600, 11.0, 2.5, 3, 1.0, (1 / 3, 1 / 3, 1 / 3), 0.3, -1.5, 4001),
    "cell_changes": (700, 13.0, 2.1, 1, 1.0, (0.8, 0.1, 0.1), 2.0, -2.0, 3000),
    "fewer_moves_than_movers": (50, 7.5, 2.5, 1, 1.0, (1 / 3, 1 / 3, 1 / 3), 0.3, -2.0, 3),
}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("config", [0, 1, 2, 3])
@pytest.mark.parametrize("case", sorted(CASES))
def test_moves_in_flight_take_the_oracles_moves(case, config, precision):
    n, L, rc, S, e, p, max_disp, lz, moves = CASES[case]
    pos = W.uniform_positions(n, L, 5)
    if e:
        side = math.ceil(n ** (1 / 3))
        k = np.arange(n)
        pos = (np.stack([k % side, k // side % side, k // side ** 2], 1) + 0.5) * (L / side)
    types = (np.arange(n) % S).astype(np.int32)
    eps, sigma = W.lorentz_berthelot([e] * S, np.linspace(1.0, 1.1, S))
    args = (*p, max_disp, 1 / 1.2, [lz] * S)
    o = O.System(L, rc, eps, sigma)
    o.build(pos, types)
    o.set_energy(o.total_energy())
    b = Box(L, rc, eps, sigma, precision=precision)
    b.set_chain_config(config)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    tol = 1e-5 if precision == "fp32" else 1e-12
    to, _ = o.run_moves(11, 0, moves, *args, tol=tol)
    _, tg = b.run_moves(11, 0, moves, Mix(*args), trace=True)
    for f in ("type", "species", "index", "accepted"):
        assert np.array_equal(tg[f], to[f]), f
    ok = np.isfinite(to["lnA"])
    assert np.all(np.abs(tg["dU"] - to["dU"])[ok] <= tol * to["uabs"][ok] + 1e-300)
    for x, y in zip(o.state(), b.get_state()[:4]):
        assert np.array_equal(x, y)
    b.check_state()
