"""GPU: particles on top of each other.  A coincident pair has U = +inf (no
pair term at eps = 0 unless coincident); a pair closer than about 6e-4 sigma has
an s^12 beyond the floats, so FP32 mode gives +inf where the value itself is
beyond them, and never NaN.

Tolerance, of the sum of |rep| + |att|: FP64 1e-12, FP32 mode 1e-10, as for
points apart."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box  # noqa: E402

TOL = {"fp64": 1e-12, "fp32": 1e-10}
FLOAT_MAX = 3.4028234e38
# distances of a trial point from its particle (the grid spacing is 2e-9)
APART = (0.0, 5e-9, 1e-7, 4e-7, 1e-6, 1e-5, 1e-4, 5e-4, 6.2e-4, 7e-4, 1e-3, 1e-2)


def _agree(got, ref, uabs, precision):
    """Within the tolerance; FP32 mode: +inf from the floats' largest value on
    (an s^12 of 8.5e37 on at eps = 1, where 4 eps s^12 passes it)."""
    assert not np.isnan(got).any()
    beyond = uabs > 0.2 * FLOAT_MAX if precision == "fp32" else np.isinf(ref)
    assert np.all(got[uabs > FLOAT_MAX] == np.inf) if precision == "fp32" else np.array_equal(np.isinf(got), np.isinf(ref))
    assert np.all(got[beyond] > 0.1 * FLOAT_MAX)
    assert np.all(np.abs(got[~beyond] - ref[~beyond]) <= TOL[precision] * uabs[~beyond])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("m", [len(APART), 40_000])
@pytest.mark.parametrize("with_abs", [False, True])
def test_trial_points_on_particles(precision, m, with_abs):
    L, n = 9.0, 300
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=2.5, n_species=1, seed=4)
    o = O.System(L, 2.5, eps, sigma)
    o.build(pos, types)
    b = Box(L, 2.5, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    tp, ts = W.insertion_points(m, L, 1, 5)
    tp = np.array(tp, np.float64)
    k = len(APART)
    at = pos[:k].copy()
    at[:, 0] = np.remainder(at[:, 0] + np.array(APART), L)
    tp[:k] = at
    got = b.trial_energy(tp, ts, with_abs=with_abs)
    got, gabs = got if with_abs else (got, None)
    pick = np.arange(min(m, 400))
    ref, uabs = o.trial_energy(tp[pick], ts[pick], with_abs=True)
    _agree(got.cpu().numpy()[pick], ref, uabs, precision)
    if with_abs:
        gabs = gabs.cpu().numpy()[pick]
        near = uabs > 0.2 * FLOAT_MAX
        assert not np.isnan(gabs).any()
        assert np.allclose(gabs[~near], uabs[~near], rtol=1e-5, atol=0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("m", [8, 40_000])
def test_no_interaction_stays_none(precision, m):
    """eps = 0: nothing however close, but for a coincident pair."""
    L = 9.0
    pos = W.uniform_positions(300, L, 3)
    b = Box(L, 2.5, [[0.0]], [[1.0]], precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.zeros(300, dtype=torch.int32))
    tp = np.array(W.insertion_points(m, L, 1, 5)[0], np.float64)
    for k, d in enumerate(APART[1:8]):
        tp[k] = pos[k]
        tp[k, 0] = np.remainder(tp[k, 0] + d, L)
    got, gabs = b.trial_energy(tp, np.zeros(m, np.int32), with_abs=True)
    assert torch.all(got == 0.0) and torch.all(gabs == 0.0)
    assert torch.all(b.trial_energy(tp, np.zeros(m, np.int32)) == 0.0)
    g = b.energy_grad()
    assert g["energy"] == 0.0 and np.isfinite(g["deps"]).all() and g["deps"][0, 0] > 0.0


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("S", [1, 3])
@pytest.mark.parametrize("apart", [1e-4, 5e-4])
def test_total_energy_and_gradient_of_an_overlap(precision, S, apart):
    L, n = 9.0, 300
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=2.5, n_species=S, seed=4)
    pos[1] = pos[0] + np.array([0.6, 0.0, 0.8]) * apart
    pos = np.remainder(pos, L)
    b = Box(L, 2.5, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    energy, g = b.total_energy(), b.energy_grad()
    if precision == "fp32":  # s^12 above 1e39
        assert energy == math.inf and g["energy"] == math.inf and g["virial"] == -math.inf
        assert not np.isnan(g["deps"]).any() and not np.isnan(g["dsigma"]).any()
    else:
        o = O.System(L, 2.5, eps, sigma)
        o.build(pos, types)
        ref = o.energy_grad()
        assert abs(energy - o.total_energy()) <= 1e-12 * abs(energy)
        for k in ("energy", "virial"):
            assert abs(g[k] - ref[k]) <= 1e-11 * abs(ref[k])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("S", [1, 3])
@pytest.mark.parametrize("steps", [0, 1, 40, 200, 2000, 50_000])
def test_gradient_of_a_pair_on_an_axis(precision, S, steps):
    """A pair `steps` grid points (2.1e-9 each) apart along x: the infinities of
    the energy, the virial and the force along x, no NaN in any result.  (A
    coincident pair's force has no direction and is not looked at.)"""
    L, n = 9.0, 300
    pos, types, eps, sigma = W.tiny_system(n=n, L=L, rc=2.5, n_species=S, seed=4)
    h = L / 2.0 ** 32
    pos[0] = (np.floor(pos[0] / h) + 0.5) * h
    pos[1] = pos[0] + np.array([steps * h, 0.0, 0.0])
    b = Box(L, 2.5, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    energy, g = b.total_energy(), b.energy_grad(input_order=True)
    force = g["dpos"].cpu().numpy()
    assert not np.isnan(g["deps"]).any() and not np.isnan(g["dsigma"]).any()
    if precision == "fp32" or steps == 0:
        assert energy == math.inf and g["energy"] == math.inf and g["virial"] == -math.inf
        assert g["deps"].max() == math.inf and g["dsigma"].max() == math.inf
    else:
        o = O.System(L, 2.5, eps, sigma)
        o.build(pos, types)
        ref = o.energy_grad()
        for k in ("energy", "virial"):
            assert abs(g[k] - ref[k]) <= 1e-11 * abs(ref[k])
    assert not np.isnan(force[2:]).any() and np.isfinite(force[2:]).all()
    if steps:
        # U falls steeply with the distance: dE/dx of the left one is +inf
        assert force[0, 0] == np.inf and force[1, 0] == -np.inf
        assert np.isfinite(force[:2, 1:]).all()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_gradient_without_interaction(precision):
    """eps = 0: no energy of a close pair, +inf of a coincident one (as the total energy)."""
    L = 9.0
    h = L / 2.0 ** 32
    pos = W.uniform_positions(300, L, 3)
    pos[0] = (np.floor(pos[0] / h) + 0.5) * h
    for steps, ref in ((40, 0.0), (0, math.inf)):
        pos[1] = pos[0] + np.array([steps * h, 0.0, 0.0])
        b = Box(L, 2.5, [[0.0]], [[1.0]], precision=precision)
        b.build_cells(torch.as_tensor(pos), torch.zeros(300, dtype=torch.int32))
        g = b.energy_grad()
        assert b.total_energy() == ref and g["energy"] == ref
        assert not np.isnan(g["deps"]).any() and g["deps"][0, 0] > 0.0
