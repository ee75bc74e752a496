"""GPU: insertions into an ideal gas of nine million particles whose acceptance
ratio lies 1e-7 from the random number, where rounding in FP32 errs by up to
2e-6: ln z + ln V just beside the midpoint between two floats (1.9e-6 apart
there), and particle counts whose logarithm rounds the other way.  Every one of
these decisions has to be taken in FP64 (rounding 1e-14)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box, Mix  # noqa: E402

L, RC, SEED, MARGIN = 100.1, 2.5, 17, 1e-7


def _moves():
    """(move, ln u) of the moves of the stream whose u lies in (0.98, 1)."""
    out = []
    for m in range(10_000):
        w = O.move_words(SEED, m)
        u = ((int(w[6]) >> 5 << 26) | (int(w[7]) >> 6)) * 2.0 ** -53
        if u > 0.98:
            out.append((m, math.log(u)))
    return out


def _cases():
    """(n, move, ln z, accepted): insertions among n particles; the FP32 value of
    ln u - ln A errs towards the wrong side by the errors of both logarithms."""
    n1 = torch.arange(9_200_000, 9_390_000, device="cuda", dtype=torch.float32)
    err = torch.log(n1).double() - torch.log(n1.double())
    moves, lnv = _moves(), math.log(L * L * L)
    out = []
    for accepted, k in ((True, int(err.argmax())), (False, int(err.argmin()))):
        n = int(n1[k]) - 1
        for m, lnu in moves:
            z = lnu + (MARGIN if accepted else -MARGIN) + math.log(n + 1)  # ln z + ln V
            lz = z - lnv
            e = float(np.float32(lz + lnv)) - (lz + lnv)
            if 0.45 * float(np.spacing(np.float32(z))) < (-e if accepted else e):
                out.append((n, m, lz, accepted))
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_close_decisions_are_taken_in_fp64(precision):
    cases = _cases()
    assert {a for *_, a in cases} == {True, False}
    side = 211  # 211^3 = 9.39e6 lattice sites
    k = torch.arange(side ** 3, device="cuda")
    sites = (torch.stack([k % side, k // side % side, k // side ** 2], 1).double() + 0.5) * (L / side)
    b = Box(L, RC, [[0.0]], [[1.0]], precision=precision, max_particles=1 << 24)
    for n, m, lz, accepted in cases:
        b.build_cells(sites[:n], torch.zeros(n, dtype=torch.int32, device="cuda"))
        _, t = b.run_moves(SEED, m, 1, Mix(0.0, 1.0, 0.0, 0.3, 1.0, [lz]), trace=True)
        assert t["type"][0] == 1 and t["dU"][0] == 0.0
        assert bool(t["accepted"][0]) == accepted, (n, m, lz)
