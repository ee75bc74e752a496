"""GPU: trial energies of a few points (one block per point) and of many
(binned by cell) against the oracle, around the line between the two: boxes
narrower than three cutoffs, cells of more records than a pass takes, an empty
box, exclusions, rejected points.

Tolerance, of the sum of |rep| + |att|: FP64 1e-12 (a few hundred roundings of
1.1e-16, six-fold in r^-12); FP32 mode 1e-10 (compensated terms to about 2^-44
each, six-fold, and as many additions in float-float)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box, Mix  # noqa: E402

TOL = {"fp64": 1e-12, "fp32": 1e-10}
FEW = 4096


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("m", [1, 2, FEW, FEW + 1, 4 * FEW, 4 * FEW + 1, 8 * FEW + 1])
@pytest.mark.parametrize("n,L,rc,S", [(0, 8.0, 2.5, 1), (90, 5.6, 2.5, 2), (1500, 7.6, 2.5, 3), (1000, 13.0, 2.5, 2)])
def test_few_and_many_points(precision, m, n, L, rc, S):
    pos, types, eps, sigma = W.tiny_system(n=max(n, 1), L=L, rc=rc, n_species=S, seed=n + 3)
    pos, types = pos[:n], types[:n]
    o = O.System(L, rc, eps, sigma)
    o.build(pos, types)
    b = Box(L, rc, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    tp, ts = W.insertion_points(m, L, S, m)
    cnt = o.counts()
    excl = np.full(m, -1, np.int64)
    if n:
        excl[::2] = (np.int64(0) << 32) | (np.arange(m)[::2] % max(1, int(cnt[0])))
    got, gabs = b.trial_energy(tp, ts, exclude=torch.as_tensor(excl), with_abs=True)
    pick = np.unique(np.concatenate([np.arange(min(m, 40)), np.arange(m)[-40:]]))
    ref, uabs = o.trial_energy(tp[pick], ts[pick], exclude=excl[pick].tolist(), with_abs=True)
    assert np.all(np.abs(got.cpu().numpy()[pick] - ref) <= TOL[precision] * uabs)
    assert np.allclose(gabs.cpu().numpy()[pick], uabs, rtol=1e-5, atol=0)
    alone = b.trial_energy(tp, ts, exclude=torch.as_tensor(excl)).cpu().numpy()
    assert np.all(np.abs(alone[pick] - ref) <= TOL[precision] * uabs)


@pytest.mark.parametrize("n,L", [(90, 5.6), (1500, 7.6), (2000, 16.0)])
def test_fp32_magnitudes_do_not_depend_on_the_path(n, L):
    """The plain FP32 sums of |rep| + |att| of the same points, one block per point
    and binned (one point more), bit for bit, also over several passes."""
    m = 8 * FEW
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=2.5, n_species=2, seed=n)
    b = Box(L, 2.5, eps, sigma, precision="fp32")
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    tp, ts = W.insertion_points(m + 1, L, 2, 6)
    excl = torch.arange(m + 1) % 11 - 1
    few = b.trial_energy(tp[:m], ts[:m], exclude=excl[:m], with_abs=True)[1]
    many = b.trial_energy(tp, ts, exclude=excl, with_abs=True)[1]
    assert torch.equal(few, many[:m])


@pytest.mark.parametrize("m", [3, FEW + 1])
def test_a_rejected_point_gets_nan_and_the_others_their_energy(m):
    L = 9.0
    pos, types, eps, sigma = W.tiny_system(n=300, L=L, rc=2.5, n_species=1, seed=4)
    b = Box(L, 2.5, eps, sigma)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    tp, ts = W.insertion_points(m, L, 1, 5)
    want = b.trial_energy(tp, ts).cpu().numpy()
    bad = torch.as_tensor(tp, dtype=torch.float64).cuda()
    bad[1, 2] = float("inf")
    sp = torch.as_tensor(ts, dtype=torch.int32).cuda()
    out = torch.zeros(m, dtype=torch.float64, device="cuda")
    assert b.trial_energy_raw(bad, sp, out) == 1  # INVALID_ARG
    got = out.cpu().numpy()
    assert np.isnan(got[1]) and np.array_equal(np.delete(got, 1), np.delete(want, 1))
    # the next call starts with a clean status
    assert np.array_equal(b.trial_energy(tp, ts).cpu().numpy(), want)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("S", [1, 2, 3, 5])
def test_forces_in_input_order(precision, S):
    """Bit for bit the species-major forces, at the input rows; refused once
    moves have changed the configuration."""
    L, n = 12.0, 700
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=2.5, n_species=S, seed=S)
    b = Box(L, 2.5, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    sm = np.argsort(types, kind="stable")
    major, rows = b.energy_grad(), b.energy_grad(input_order=True)
    assert np.array_equal(rows["dpos"].cpu().numpy()[sm], major["dpos"].cpu().numpy())
    for k in ("energy", "virial"):
        assert rows[k] == major[k]
    b.run_moves(1, 0, 10, Mix(0.4, 0.3, 0.3, 0.3, 1.0, [-2.0] * S))
    with pytest.raises(RuntimeError):
        b.energy_grad(input_order=True)

