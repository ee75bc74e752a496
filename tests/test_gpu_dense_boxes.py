"""GPU: total energy and gradient against the oracle where a neighbourhood takes
several passes or none: cells of more particles than a chunk, more records than
a pass holds, rows with a remainder, boxes narrower than three cutoffs, three
and five species, one particle.

Tolerances: the energy to 1e-12 (FP64) or 1e-10 (FP32 mode, compensated) of the
sum of |rep| + |att|; the gradient, of its largest component (whose terms add to
a few times it), FP64 4e-7 (forces are stored in FP32), FP32 mode 6e-6 (a term
carries about 25 roundings of 6e-8: r^-2 to 1.5e-7, r^-12 six-fold).  Energy and
virial of the gradient the same, of the sum."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle as O  # noqa: E402
from paper_1408_3764_gb300 import workloads as W  # noqa: E402
from paper_1408_3764_gb300.gcmc import Box  # noqa: E402


def _lattice(n, L, seed):
    """n sites of a cubic lattice, displaced by up to 0.15 of its spacing."""
    rng = np.random.default_rng(seed)
    side = int(np.ceil(n ** (1 / 3) - 1e-9))
    site = rng.permutation(side ** 3)[:n]
    ijk = np.stack([site % side, site // side % side, site // side ** 2], 1)
    return ((ijk + 0.5 + rng.uniform(-0.15, 0.15, (n, 3))) * (L / side)) % L


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n,L,rc,S", [(1, 6.0, 2.5, 1), (33, 5.6, 2.5, 2), (700, 5.6, 2.5, 1), (2197, 7.6, 2.5, 3),
                                      (1331, 10.1, 2.5, 5), (3000, 13.0, 4.0, 2)])
def test_energy_and_gradient(precision, n, L, rc, S):
    _, types, eps, sigma = W.tiny_system(n=n, L=L, rc=rc, n_species=S, seed=n)
    pos = _lattice(n, L, n)
    o = O.System(L, rc, eps, sigma)
    o.build(pos, types)
    b = Box(L, rc, eps, sigma, precision=precision)
    b.build_cells(torch.as_tensor(pos), torch.as_tensor(types))
    order = np.argsort(types, kind="stable")
    first = np.concatenate([[0], np.cumsum(o.counts())])
    excl = [(int(types[p]) << 32) | int(r - first[types[p]]) for r, p in enumerate(order)]
    scale = 0.5 * o.trial_energy(pos[order], types[order], exclude=excl, with_abs=True)[1].sum()
    assert abs(b.total_energy() - o.total_energy()) <= (1e-12 if precision == "fp64" else 1e-10) * scale
    got, ref, tol = b.energy_grad(), o.energy_grad(), 4e-7 if precision == "fp64" else 6e-6
    for k in ("dpos", "deps", "dsigma"):
        x = got[k].cpu().numpy() if k == "dpos" else got[k]
        assert np.all(np.abs(x - ref[k]) <= tol * np.abs(ref[k]).max() + 1e-300), k
    assert abs(got["energy"] - ref["energy"]) <= tol * scale
    assert abs(got["virial"] - ref["virial"]) <= 12 * tol * scale
