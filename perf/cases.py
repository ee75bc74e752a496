"""The work that users of the library have it do, as cases that can be timed
and checked: trial energies, cell build with full-system energy, the
differentiable energy, GCMC chains (one box, a batch of boxes, the microcell
list).  Sizes follow the workloads of ``paper_1408_3764_gb300.workloads``.

A case is a dict of plain values; ``kind`` says which entry point it goes
through and the other keys are its sizes and options.
"""
import math

import numpy as np
import torch

from paper_1408_3764_gb300 import Batch, Box, Mix, cell_list_energy

GRID = 4294967296.0
# ln z along the T* = 1.2 isotherm (the table of the workloads module)
RHO_TABLE = (0.1, 0.2, 0.3, 0.4, 0.5, 0.6, 0.7)
LOGZ_TABLE = (-2.927, -2.788, -2.726, -2.752, -2.711, -2.351, -1.964)


def listed():
    one = dict(rho=0.6, rc=3.0, species=1, temperature=1.5)
    mix = dict(rho=0.7, rc=3.0, species=2, temperature=1.3)
    return [
        # Widom probes between blocks of a small plain run: a call of a few
        # microseconds of arithmetic, where launches and the wait count
        dict(name="trial_64_fp64", kind="trial", n=2048, m=64, precision="fp64", exclude=False, with_abs=False,
             rho=0.5, rc=2.5, species=1, temperature=1.2),
        # chemical potential of the million-particle mixture: one batch of insertions
        dict(name="trial_1m_mixture_fp32", kind="trial", n=1 << 20, m=1_000_000, precision="fp32", exclude=False,
             with_abs=False, **mix),
        # energies of particles in place (each excluding itself) with their
        # error scales, as the reference of a precision check: FP64, odd count
        dict(name="trial_50001_self_fp64", kind="trial", n=131072, m=50_001, precision="fp64", exclude=True,
             with_abs=True, **one),
        # a new configuration of the million-particle mixture: binned, total energy
        dict(name="energy_1m_mixture_fp32", kind="energy", n=1 << 20, precision="fp32", **mix),
        # the cutoff-sweep box in FP64, as a check of a running energy
        dict(name="energy_87296_fp64", kind="energy", n=87296, precision="fp64", rho=0.666, rc=3.25, species=1,
             temperature=1.5),
        # force-field fitting step on the mixture: energy and all its gradients
        dict(name="grad_262k_mixture_fp32", kind="grad", n=1 << 18, precision="fp32", rho=0.65, rc=3.0, species=2,
             temperature=1.3),
        # the same on a small three-species training sample in FP64
        dict(name="grad_6001_three_species_fp64", kind="grad", n=6001, precision="fp64", rho=0.6, rc=2.5, species=3,
             temperature=1.3),
        # plain GCMC of the 2,048-particle fluid
        dict(name="chain_2048_fp64", kind="chain", n=2048, moves=10_000, precision="fp64", virial=False, rho=0.5,
             rc=2.5, species=1, temperature=1.2, log_z0=-2.786),
        # one large box in FP32 mode
        dict(name="chain_131072_fp32", kind="chain", n=131072, moves=20_000, precision="fp32", virial=False,
             log_z0=-1.405, **one),
        # a mixture whose pressure is averaged along the chain; odd sizes
        dict(name="chain_mixture_virial_fp32", kind="chain", n=4001, moves=9_999, precision="fp32", virial=True,
             rho=0.65, rc=3.0, species=2, temperature=1.3, log_z0=-1.193, log_z1=-1.086),
        # the batched isotherm, whole step: bin and total energy, moves, forces, export
        dict(name="isotherm_64_fp32", kind="isotherm", chains=64, n_min=500, n_max=20_000, rho_min=0.1, rho_max=0.7,
             moves=100_000, precision="fp32", rc=2.5, temperature=1.2),
        # the microcell list on the cutoff-sweep box
        dict(name="micro_87296_fp32", kind="micro", n=87296, moves=4_000, precision="fp32", rho=0.666, rc=2.5,
             species=1, temperature=1.5, log_z0=-0.644),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["trial", "trial", "energy", "grad", "chain", "chain", "isotherm", "micro"])
    precision = rng.choice(["fp32", "fp64"])
    if kind == "isotherm":
        n_max = logint(2_000, 20_000)
        return dict(kind=kind, chains=logint(4, 64), n_min=500, n_max=n_max, rho_min=0.1,
                    rho_max=round(rng.uniform(0.3, 0.7), 3), moves=logint(2_000, 40_000), precision=precision, rc=2.5,
                    temperature=1.2)
    rho = round(rng.uniform(0.1, 0.7), 3)
    n_hi = {"trial": 1 << 20, "energy": 1 << 20, "grad": 1 << 18, "chain": 131072, "micro": 87296}[kind]
    n = logint(500, n_hi)
    if kind in ("chain", "micro"):  # the chain keeps its cell counts on chip: boxes up to about 60 sigma
        rho = round(max(rho, n / 60.0 ** 3), 3)
    edge = (n / rho) ** (1.0 / 3.0)
    case = dict(kind=kind, n=n, precision=precision, rho=rho,
                rc=round(min(rng.uniform(2.5, 4.25 if kind != "trial" else 3.5), 0.499 * edge), 3),
                species=rng.choice([1, 1, 2, 3]), temperature=round(rng.uniform(1.2, 1.5), 3))
    if kind == "trial":
        case.update(m=logint(1, 1_000_000), exclude=rng.random() < 0.5, with_abs=rng.random() < 0.5)
    if kind in ("chain", "micro"):
        lz = float(np.interp(rho, RHO_TABLE, LOGZ_TABLE))
        case.update(moves=logint(500, 20_000 if kind == "chain" else 4_000))
        case.update({"log_z%d" % s: round(lz - math.log(case["species"]), 3) for s in range(case["species"])})
    if kind == "chain":
        case.update(virial=rng.random() < 0.3)
    return case


# ------------------------------------------------------------------ inputs ---

def _edge(n, rho):
    return float((n / rho) ** (1.0 / 3.0))


def _fields(species):
    """Lorentz-Berthelot tables of 1 to 3 species (sigma 1 to 1.2, eps 1 to 0.8)."""
    s = np.array([1.0, 1.2, 1.1])[:species]
    e = np.array([1.0, 0.8, 0.9])[:species]
    return np.sqrt(np.outer(e, e)), 0.5 * (s[:, None] + s[None, :])


def _fluid(n, L, species, seed):
    """n particles without deep overlaps: sites of a cubic lattice taken at
    random and displaced; 80 % of them species 0.  [n, 3] FP64 and [n] int32
    (CPU)."""
    g = torch.Generator().manual_seed(int(seed) * 1_000_003 + 17)
    side = max(1, int(math.ceil(n ** (1.0 / 3.0) - 1e-9)))
    while side ** 3 < n:
        side += 1
    site = torch.randperm(side ** 3, generator=g)[:n]
    ijk = torch.stack([site % side, (site // side) % side, site // (side * side)], 1).to(torch.float64)
    jit = (torch.rand((n, 3), generator=g, dtype=torch.float64) - 0.5) * 0.3
    pos = torch.remainder((ijk + 0.5 + jit) * (L / side), L)
    u = torch.rand(n, generator=g)
    types = torch.zeros(n, dtype=torch.int32)
    for s in range(1, species):
        types[u > 0.8 + 0.2 * (s - 1) / max(1, species - 1)] = s
    return pos, types


def _trial_points(case, L, seed, types):
    """Trial points: uniform insertions, or (exclude) displaced particles with
    the ids they leave out.  CPU tensors."""
    g = torch.Generator().manual_seed(int(seed) * 7_919 + 3)
    m = case["m"]
    if not case["exclude"]:
        pos = torch.rand((m, 3), generator=g, dtype=torch.float64) * L
        return pos, torch.randint(0, case["species"], (m,), generator=g, dtype=torch.int32), None
    pick = torch.randint(0, case["n"], (m,), generator=g)
    rank = torch.zeros(case["n"], dtype=torch.int64)  # index of a particle within its species
    for s in range(case["species"]):
        w = types == s
        rank[w] = torch.arange(int(w.sum()))
    step = (torch.rand((m, 3), generator=g, dtype=torch.float64) - 0.5) * 0.1
    sp = types[pick]
    return (pick, step), sp, (sp.to(torch.int64) << 32) | rank[pick]


def _isotherm(case, seed):
    """(n, L, ln z, seed) of each chain: N0 log-uniform (the case's own), rho linear."""
    rng = np.random.default_rng(4)
    K = case["chains"]
    ns = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), K)).astype(np.int64)
    rhos = np.linspace(case["rho_min"], case["rho_max"], K)
    return [(int(n), max(_edge(int(n), float(r)), 2.001 * case["rc"]),
             float(np.interp(r, RHO_TABLE, LOGZ_TABLE)), 1000 + 64 * int(seed) + k)
            for k, (n, r) in enumerate(zip(ns, rhos))]


def _log_z(case):
    return [case["log_z%d" % s] for s in range(case["species"])]


def _rows(L):
    """Rows that hold any configuration of a box (the fluid stays below rho 0.95)."""
    return int(0.95 * L ** 3) + 512


def _buffers(rows, device):
    return (torch.zeros((rows, 3), dtype=torch.float64, device=device),
            torch.zeros(rows, dtype=torch.int32, device=device))


def _mix(case, log_z, virial=False):
    third = 1.0 / 3.0
    return Mix(third, third, third, 0.3, 1.0 / case["temperature"], list(log_z), virial=virial)


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "isotherm":
        st = dict(case=case, boxes=[], pos=[], types=[], mixes=[], seeds=[])
        eps, sigma = _fields(1)
        rows = []
        for n, L, lz, sd in _isotherm(case, seed):
            pos, types = _fluid(n, L, 1, sd)
            st["boxes"].append(Box(L, case["rc"], eps, sigma, precision=case["precision"]))
            st["pos"].append(pos.to(dev))
            st["types"].append(types.to(dev))
            st["mixes"].append(_mix(case, [lz]))
            st["seeds"].append(sd)
            rows.append(_rows(L))
        st["batch"] = Batch(st["boxes"])
        # forces and final configurations of all chains, one after another
        st["all"] = _buffers(sum(rows), dev) + (torch.zeros((sum(rows), 3), dtype=torch.float32, device=dev),)
        st["out_pos"], st["out_types"], st["dpos"] = (list(torch.split(t, rows)) for t in st["all"])
        return st
    L = _edge(case["n"], case["rho"])
    eps, sigma = _fields(case["species"])
    pos, types = _fluid(case["n"], L, case["species"], seed)
    st = dict(case=case, L=L, seed=int(seed), types=types.to(dev))
    if case["kind"] == "grad":
        st.update(pos=pos.to(dev, torch.float32), eps=torch.tensor(eps), sigma=torch.tensor(sigma))
        return st
    st["pos"] = pos.to(dev)
    box = st["box"] = Box(L, case["rc"], eps, sigma, precision=case["precision"])
    if case["kind"] == "trial":
        box.build_cells(st["pos"], st["types"])
        pts, sp, ex = _trial_points(case, L, seed, types)
        if ex is not None:
            pts = torch.remainder(pos[pts[0]] + pts[1], L)
            ex = ex.to(dev)
        st.update(points=pts.to(dev), sp=sp.to(dev), exclude=ex)
    elif case["kind"] in ("chain", "micro"):
        st["mix"] = _mix(case, _log_z(case), case.get("virial", False))
        st["out_pos"], st["out_types"] = _buffers(_rows(L), dev)
        if case["kind"] == "micro":
            box.build_cells(st["pos"], st["types"]).build_microcells(1.0)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "trial":
        return st["box"].trial_energy(st["points"], st["sp"], st["exclude"], with_abs=case["with_abs"])
    if kind == "energy":
        box = st["box"].build_cells(st["pos"], st["types"])
        return [box.total_energy(), *box.cell_list()]
    if kind == "grad":
        pos = st["pos"].detach().requires_grad_(True)
        eps = st["eps"].detach().requires_grad_(True)
        sigma = st["sigma"].detach().requires_grad_(True)
        e = cell_list_energy(pos, eps, sigma, st["types"], st["L"], case["rc"], case["precision"])
        return [e.detach(), *torch.autograd.grad(e, [pos, eps, sigma])]
    if kind == "isotherm":
        batch = st["batch"]
        e0 = batch.prepare(st["pos"], st["types"])
        stats = batch.run_moves(st["seeds"], 0, case["moves"], st["mixes"])
        e1, w1 = batch.energy_grad(st["dpos"])
        n = batch.export_positions(st["out_pos"], st["out_types"])
        stats = [_stats(s) for s in stats]
        return dict(start_energy=e0, end_energy=e1, end_virial=w1, counts=n, pos=st["all"][0], types=st["all"][1],
                    dpos=st["all"][2], **{k: np.array([s[k] for s in stats]) for k in stats[0]})
    box = st["box"].build_cells(st["pos"], st["types"])
    if kind == "micro":
        stats = box.run_moves_micro(st["seed"], 0, case["moves"], st["mix"])
    else:
        stats = box.run_moves(st["seed"], 0, case["moves"], st["mix"])
    box.export_positions(st["out_pos"], st["out_types"])
    return dict(pos=st["out_pos"], types=st["out_types"], **_stats(stats))


def _stats(s):
    """The results of a run (its device time left out)."""
    out = dict(attempted=np.array(s["attempted"], np.int64), accepted=np.array(s["accepted"], np.int64),
               n_species=np.array(s["n"], np.int64), moves_done=s["moves_done"], energy=s["energy"],
               sum_energy=s["sum_energy"], sum_n=s["sum_n"])
    if not math.isnan(s["virial"]):
        out.update(virial=s["virial"], sum_virial=s["sum_virial"])
    return out


def work(case):
    """Bytes: inputs read once, outputs written once.  Operations: 20 per pair
    inside the cutoff for an energy, 30 with its gradient; a displacement
    evaluates two positions, an insertion or deletion one."""
    sphere = 4.0 / 3.0 * math.pi * case["rc"] ** 3
    if case["kind"] == "isotherm":
        K = case["chains"]
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        n = K * (case["n_max"] - case["n_min"]) / (hi - lo)  # mean of the log-uniform N0
        near = 0.5 * (case["rho_min"] + case["rho_max"]) * sphere
        return dict(bytes=n * (28 + 28 + 12), flops=n * near / 2 * (20 + 30) + K * case["moves"] * 4 / 3 * near * 20)
    n, near = case["n"], case["rho"] * sphere
    if case["kind"] == "trial":
        per = 24 + 4 + 8 + (8 if case["exclude"] else 0) + (8 if case["with_abs"] else 0)
        return dict(bytes=16.0 * n + per * case["m"], flops=case["m"] * near * 20)
    if case["kind"] == "energy":
        return dict(bytes=32.0 * n + 8.0 * max(3, int(_edge(n, case["rho"]) // case["rc"])) ** 3, flops=n * near / 2 * 20)
    if case["kind"] == "grad":
        return dict(bytes=28.0 * n, flops=n * near / 2 * 30)
    return dict(bytes=56.0 * n, flops=n * near / 2 * 20 + case["moves"] * 4 / 3 * near * 20)


# ------------------------------------------------- the same in 64 bits ------
# Positions are the documented grid points (2^32 per edge), as plain integers;
# everything below is torch and numpy in 64 bits.

def _grid(pos, L):
    return torch.floor(pos.to(torch.float64) * (GRID / L)).to(torch.int64) & 0xFFFFFFFF


def _wrap(d):
    return ((d + 0x80000000) & 0xFFFFFFFF) - 0x80000000


class _Neighbours:
    """Particles in cells of edge >= rc, padded, for gathering the 27 around a point."""

    def __init__(self, X, types, L, rc):
        self.T = max(3, int(L // rc))
        self.X, self.types = X, types
        self.L, self.rc = L, rc
        cell = self.cell(X)
        order = torch.argsort(cell, stable=True)
        count = torch.bincount(cell, minlength=self.T ** 3)
        start = torch.cumsum(count, 0) - count
        self.cap = int(count.max()) if len(X) else 1
        self.table = torch.full((self.T ** 3, self.cap), -1, dtype=torch.int64, device=X.device)
        slot = torch.arange(len(X), device=X.device) - start[cell[order]]
        self.table[cell[order], slot] = order

    def coords(self, X):
        return (X * self.T) >> 32

    def cell(self, X):
        c = self.coords(X)
        return (c[:, 2] * self.T + c[:, 1]) * self.T + c[:, 0]

    def pairs(self, P, sp, own, eps, sigma, chunk=1 << 15):
        """Per chunk of points: (slice, partner index, separation in length
        units [c, k, 3], r^2, rep, att) with zeros outside the cutoff."""
        o = torch.arange(-1, 2, device=P.device)
        off = torch.cartesian_prod(o, o, o)
        h = self.L / GRID
        r2max = math.ceil((self.rc * (GRID / self.L)) ** 2)
        for a in range(0, len(P), chunk):
            sl = slice(a, min(len(P), a + chunk))
            c = (self.coords(P[sl])[:, None, :] + off[None]) % self.T
            j = self.table[(c[..., 2] * self.T + c[..., 1]) * self.T + c[..., 0]].flatten(1)
            d = _wrap(P[sl][:, None, :] - self.X[j.clamp(min=0)])
            df = d.to(torch.float64)
            g2 = (df * df).sum(-1)
            near = (g2 < 1.001 * r2max) & (j >= 0) & (j != own[sl][:, None])
            exact2 = (d * d).sum(-1)  # below 2^63 inside and near the cutoff
            near &= exact2 < r2max
            r2 = torch.where(near, g2 * (h * h), torch.ones_like(g2))
            e = eps[sp[sl].long()[:, None], self.types[j.clamp(min=0)].long()]
            s = sigma[sp[sl].long()[:, None], self.types[j.clamp(min=0)].long()]
            s6 = (s * s / r2) ** 3
            zero = torch.zeros_like(r2)
            yield sl, j, df * h, r2, torch.where(near, 4 * e * s6 * s6, zero), torch.where(near, 4 * e * s6, zero)


def exact(case, seed):
    kind = case["kind"]
    if kind == "isotherm":
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    L = _edge(case["n"], case["rho"])
    eps_n, sigma_n = _fields(case["species"])
    pos, types = _fluid(case["n"], L, case["species"], seed)
    if kind == "grad":
        pos = pos.to(torch.float32).to(torch.float64)
    X, t = _grid(pos, L).to(dev), types.to(dev)
    eps, sigma = torch.tensor(eps_n, device=dev), torch.tensor(sigma_n, device=dev)
    nb = _Neighbours(X, t, L, case["rc"])
    ids = torch.arange(case["n"], device=dev)
    chunk = max(256, (1 << 24) // (27 * nb.cap))
    if kind == "trial":
        pts, sp, ex = _trial_points(case, L, seed, types)
        own = torch.full((case["m"],), -2, dtype=torch.int64, device=dev)
        if ex is not None:
            own = pts[0].to(dev)
            pts = torch.remainder(pos[pts[0]] + pts[1], L)
        e = torch.zeros(case["m"], dtype=torch.float64, device=dev)
        a = torch.zeros_like(e)
        for sl, _, _, _, rep, att in nb.pairs(_grid(pts, L).to(dev), sp.to(dev), own, eps, sigma, chunk):
            e[sl] = (rep - att).sum(1)
            a[sl] = (rep + att).sum(1)
        return (e, a) if case["with_abs"] else e
    if kind == "grad":
        S = case["species"]
        E = torch.zeros((), dtype=torch.float64, device=dev)
        F = torch.zeros((case["n"], 3), dtype=torch.float64, device=dev)
        de = torch.zeros(S * S, dtype=torch.float64, device=dev)
        ds = torch.zeros_like(de)
        for sl, j, d, r2, rep, att in nb.pairs(X, t, ids, eps, sigma, chunk):
            E += 0.5 * (rep - att).sum()
            F[sl] = ((-12 * rep + 6 * att) / r2)[..., None].mul(d).sum(1)
            k = t[sl].long()[:, None] * S + t[j.clamp(min=0)].long()
            safe = eps.flatten()[k]
            de += 0.5 * torch.bincount(k.flatten(), ((rep - att) / safe).flatten(), minlength=S * S)
            ds += 0.5 * torch.bincount(k.flatten(), ((12 * rep - 6 * att) / sigma.flatten()[k]).flatten(),
                                       minlength=S * S)
        return [E, F, de.reshape(S, S).cpu(), ds.reshape(S, S).cpu()]
    E = W = 0.0
    for _, _, _, _, rep, att in nb.pairs(X, t, ids, eps, sigma, chunk):
        E += 0.5 * float((rep - att).sum())
        W += 0.5 * float((6 * att - 12 * rep).sum())
    if kind == "energy":
        cell = nb.cell(X)
        count = torch.bincount(cell, minlength=nb.T ** 3)
        return [E, (torch.cumsum(count, 0) - count).to(torch.int32), count.to(torch.int32),
                torch.argsort(cell, stable=True).to(torch.int32)]
    return _exact_chain(case, seed, L, X.cpu().numpy(), types.numpy(), eps_n, sigma_n, E, W)


def _philox(counters, key):
    """Philox4x32-10 (Salmon et al., SC'11) on [4, k] uint64 counters."""
    c = [x.astype(np.uint64) for x in counters]
    k0, k1, low = int(key) & 0xFFFFFFFF, (int(key) >> 32) & 0xFFFFFFFF, np.uint64(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & low,
             (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _pick(n, w, deletion):
    """The documented choice among n candidates: rejection over the next power of two."""
    k = (n - 1).bit_length()
    if k == 0:
        return 0
    tries = [w[1] >> (32 - k)]
    if deletion:
        tries += [w[2] >> (32 - k), w[3] >> (32 - k)]
    elif k <= 16:
        tries.append(((w[1] << 16) & 0xFFFFFFFF) >> (32 - k))
    for d in tries:
        if d < n:
            return d
    return ((w[4] if deletion else w[5]) * n) >> 32


def _exact_chain(case, seed, L, X0, types, eps, sigma, E, W):
    S, moves, rc = case["species"], case["moves"], case["rc"]
    beta, q, log_z = 1.0 / case["temperature"], GRID / L, _log_z(case)
    h2, r2max, T = (L / GRID) ** 2, math.ceil((rc * q) ** 2), max(3, int(L // rc))
    m = np.arange(moves, dtype=np.uint64)
    zero = np.zeros(moves, np.uint64)
    words = np.stack(_philox([m, zero, zero, zero], seed) + _philox([m, zero, zero, zero + np.uint64(1)], seed), 1)
    words = words.astype(np.int64).tolist()
    room = case["n"] + moves + 1
    X = np.zeros((room, 3), np.int64)
    X[: case["n"]] = X0
    sp = np.zeros(room, np.int64)
    sp[: case["n"]] = types
    ids = [np.flatnonzero(types == s).tolist() for s in range(S)]  # rows of each species by index
    cells = [[] for _ in range(T ** 3)]
    xt = (X0 * T) >> 32
    for i, c in enumerate(((xt[:, 2] * T + xt[:, 1]) * T + xt[:, 0]).tolist()):
        cells[c].append(i)
    around = [[(k - 1) % T, k, (k + 1) % T] for k in range(T)]

    def cell(p):
        return (((p[2] * T) >> 32) * T + ((p[1] * T) >> 32)) * T + ((p[0] * T) >> 32)

    def energy(p, s, own):
        rows = []
        for z in around[(p[2] * T) >> 32]:
            for y in around[(p[1] * T) >> 32]:
                for x in around[(p[0] * T) >> 32]:
                    rows += cells[(z * T + y) * T + x]
        j = np.array(rows, np.int64)
        d = _wrap(X[j] - np.array(p, np.int64))
        near = (np.abs(d).max(1, initial=0) <= math.isqrt(r2max) + 1) & (j != own)
        d, j = d[near], j[near]
        g2 = (d * d).sum(1)
        keep = g2 < r2max
        g2, j = g2[keep].astype(np.float64), j[keep]
        if (g2 == 0).any():
            return math.inf, math.inf
        e, sg = eps[s, sp[j]], sigma[s, sp[j]]
        s6 = (sg * sg / (g2 * h2)) ** 3
        return float((4 * e * (s6 * s6 - s6)).sum()), float((4 * e * (6 * s6 - 12 * s6 * s6)).sum())

    D = int(0.3 * q)
    thr0, thr1 = int((1.0 / 3.0) * GRID), int((1.0 / 3.0 + 1.0 / 3.0) * GRID)
    lnV = math.log(L * L * L)
    free, att, acc = case["n"], [0, 0, 0], [0, 0, 0]
    sumE = sumW = 0.0
    sumN = 0
    for w in words:
        kind = 0 if w[0] < thr0 else (1 if w[0] < thr1 else 2)
        att[kind] += 1
        s, i, dU, dW, lnK = 0, -1, math.inf, 0.0, 0.0
        total = sum(len(x) for x in ids)
        if kind == 0 and total:
            i = _pick(total, w, False)
            while i >= len(ids[s]):
                i -= len(ids[s])
                s += 1
            row = ids[s][i]
            old = X[row].tolist()
            new = [(old[a] + ((w[2 + a] * (2 * D + 1)) >> 32) - D) & 0xFFFFFFFF for a in range(3)]
            e0, w0 = energy(old, s, row)
            e1, w1 = energy(new, s, row)
            dU, dW = e1 - e0, w1 - w0
        elif kind:
            s = (w[5] * S) >> 32
            n = len(ids[s])
            if kind == 1:
                new = w[2:5]
                dU, dW = energy(new, s, -1)
                lnK = log_z[s] + lnV - math.log(n + 1)
            elif n:
                i = _pick(n, w, True)
                row = ids[s][i]
                old = X[row].tolist()
                dU, dW = (-v for v in energy(old, s, row))
                lnK = math.log(n) - log_z[s] - lnV
        u = (((w[6] >> 5) << 26) | (w[7] >> 6)) * 2.0 ** -53
        if dU != math.inf and (u == 0.0 or math.log(u) < lnK - beta * dU):
            acc[kind] += 1
            E += dU
            W += dW
            if kind != 1:
                cells[cell(old)].remove(row)
            if kind == 2:
                last = ids[s].pop()
                if i < len(ids[s]):
                    ids[s][i] = last
            else:
                if kind == 1:
                    row, free = free, free + 1
                    sp[row] = s
                    ids[s].append(row)
                X[row] = new
                cells[cell(new)].append(row)
        sumE += E
        sumW += W
        sumN += sum(len(x) for x in ids)
    stats = dict(attempted=np.array(att, np.int64), accepted=np.array(acc, np.int64),
                 n_species=np.array([len(x) for x in ids], np.int64), moves_done=moves, energy=E, sum_energy=sumE,
                 sum_n=float(sumN))
    if case.get("virial"):
        stats.update(virial=W, sum_virial=sumW)
    rows = [r for x in ids for r in x]
    pos, out_types = _buffers(_rows(L), "cpu")
    pos[: len(rows)] = torch.tensor((X[rows].astype(np.float64) + 0.5) * (L / GRID))
    out_types[: len(rows)] = torch.tensor(sp[rows].astype(np.int32))
    return dict(pos=pos, types=out_types, **stats)
