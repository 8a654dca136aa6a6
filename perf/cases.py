"""What GMP featurization is measured on: the calls a user of the package makes.

Structures are synthetic and seeded.  The probe sets, element tables and
sizes of the listed cases are those of this repository's own workloads
(`synth.py`: the 64-atom box, the 4,096-atom FCC crystal, batches of small
structures, the alloy slab, the perfect crystal); `draw` takes other sizes,
orders, widths, cutoffs and tables of the same kinds.
"""
import itertools
import math

import numpy as np
import torch

from paper_2303_12980_gb300 import synth
from paper_2303_12980_gb300.binding import GMPFeaturizer

# Probe sets: the highest order, the number of sigmas and their range, the
# cutoff, and the element table (elements, Gaussians per element).
BOX = dict(lmax=2, density=False, n_sigma=4, s_lo=0.1, s_hi=1.0, cutoff=6.0, n_el=2, n_gauss=4)
CRYSTAL = dict(lmax=4, density=False, n_sigma=8, s_lo=0.05, s_hi=1.2, cutoff=8.0, n_el=3, n_gauss=5)
BATCH = dict(lmax=4, density=False, n_sigma=8, s_lo=0.05, s_hi=1.2, cutoff=7.0, n_el=10, n_gauss=5)
SLAB = dict(lmax=6, density=False, n_sigma=16, s_lo=0.05, s_hi=1.5, cutoff=8.0, n_el=6, n_gauss=6)


def _fcc(nx, ny, nz, a, jitter, vacancies=0, vacuum=0.0):
    return dict(system="fcc", nx=nx, ny=ny, nz=nz, a=a, jitter=jitter, vacancies=vacancies, vacuum=vacuum)


def listed():
    return [
        # one small molecule-sized box, featurized by itself: interactive use,
        # a descriptor for one structure; latency and launches are what counts
        dict(name="box64_features", call="features", system="box", atoms=64, **BOX),
        # the same box inside molecular dynamics with a feature-based energy:
        # features and forces each step
        dict(name="box64_vjp", call="vjp", system="box", atoms=64, **BOX),
        # a crystal supercell of ordinary size: descriptors of every site
        dict(name="crystal4096_features", call="features", **_fcc(8, 8, 16, 3.6, 0.1), **CRYSTAL),
        # forces on it
        dict(name="crystal4096_vjp", call="vjp", **_fcc(8, 8, 16, 3.6, 0.1), **CRYSTAL),
        # its feature primes: the derivatives of every feature of every site
        # with respect to every neighbor's position, kept for fitting
        dict(name="crystal4096_jacobian", call="jacobian", **_fcc(8, 8, 16, 3.6, 0.1), **CRYSTAL),
        # features on a grid of points of the crystal (a density or a map is
        # fitted to them), the local density among the features; odd counts
        dict(name="crystal3999_points", call="points", points=10007, **_fcc(10, 10, 10, 3.6, 0.1, vacancies=1),
             **dict(CRYSTAL, density=True)),
        # a training step's energies and forces on a batch of 10,000
        # molecules, clusters and small cells (8 to 256 atoms), launch shapes
        # tuned once as a long training run does
        dict(name="batch10k_vjp", call="vjp", system="batch", structures=10000, tuned=True, **BATCH),
        # inference on a batch of such structures
        dict(name="batch2500_features", call="features", system="batch", structures=2500, **BATCH),
        # a dataset passed through one handle in minibatches, each of them new
        # to it: structures are read, featurized and written out
        dict(name="screen_features", call="screen", system="batch", structures=100, minibatches=8, **BATCH),
        # the largest: features and forces of an alloy slab of 262,144 atoms,
        # orders 0-6, 16 sigmas, launch shapes tuned once
        dict(name="slab262k_vjp", call="vjp", tuned=True, **_fcc(32, 32, 64, 3.9, 0.15, vacuum=62.4), **SLAB),
        # a smaller slab with vacancies, forces and stress for cell relaxation
        dict(name="slab32k_virial", call="virial", **_fcc(16, 16, 32, 3.9, 0.15, vacancies=21, vacuum=62.4), **SLAB),
        # a perfect one-element crystal, as structure databases hold them: the
        # symmetric sites make features cancel, which have to be refined
        dict(name="perfect32k_features", call="features", **_fcc(16, 16, 32, 3.9, 0.0), **dict(SLAB, n_el=1)),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["features", "features", "vjp", "vjp", "vjp", "jacobian", "points", "screen", "virial"])
    s_lo = round(_log(rng, 0.05, 0.2), 3)
    probe = dict(lmax=rng.choice([1, 2, 3, 4, 5, 6]), density=rng.random() < 0.3, n_sigma=rng.choice([3, 4, 6, 8, 10, 12, 16, 18]),
                 s_lo=s_lo, s_hi=round(s_lo * _log(rng, 6.0, 20.0), 3), cutoff=round(rng.uniform(5.0, 8.0), 2),
                 n_el=rng.randint(1, 8), n_gauss=rng.randint(3, 8))
    big = 100_000 if call in ("features", "vjp") else 30_000
    if call == "jacobian":
        big = 4000  # dense rows: megabytes per hundred atoms
    system = "batch" if call == "screen" else rng.choice(["box", "fcc", "fcc", "batch"])
    if system == "box":
        c = dict(system="box", atoms=int(_log(rng, 9, 400)))
    elif system == "fcc":
        cells = max(8.0, _log(rng, 200, big) / 4)
        nx = max(2, round(cells ** (1 / 3) * rng.uniform(0.7, 1.1)))
        ny = max(2, round(cells ** (1 / 3) * rng.uniform(0.7, 1.1)))
        nz = max(2, int(cells / (nx * ny)))
        c = _fcc(nx, ny, nz, round(rng.uniform(3.5, 4.3), 2), rng.choice([0.0, 0.05, 0.1, 0.15]), vacancies=rng.randint(0, 5),
                 vacuum=rng.choice([0.0, 0.0, 20.0]))
    else:
        c = dict(system="batch", structures=int(_log(rng, 10, max(20, big / 72))))
    if call == "points":
        c["points"] = int(_log(rng, 100, 30000))
    if call == "screen":
        c["structures"] = int(_log(rng, 10, 200))
        c["minibatches"] = rng.randint(2, 9)
    return dict(call=call, **c, **probe)


# ------------------------------------------------------------------- inputs
def _orders(case):
    return ([-1] if case["density"] else []) + list(range(case["lmax"] + 1))


def _sigmas(case):
    return [float(s) for s in np.geomspace(case["s_lo"], case["s_hi"], case["n_sigma"])]


def _table(case):
    """Element tables belong to the probe set, not to the structures: the
    same ones for every seed."""
    rng = np.random.default_rng(1000)
    charges = rng.integers(1, 9, case["n_el"])
    return synth.gaussian_table(rng, charges, case["n_gauss"])


def _cube(rng, n):
    """n atoms in a periodic cube at 0.08 atoms/A^3, at least 1 A apart: random
    sites of a cubic grid, displaced within the room that leaves."""
    L = (n / 0.08) ** (1 / 3)
    m = math.ceil(round(n ** (1 / 3), 9))
    a = L / m
    at = rng.permutation(m ** 3)[:n]
    site = np.stack([at // (m * m), at // m % m, at % m], 1) + 0.5
    return site * a + rng.uniform(-0.5, 0.5, (n, 3)) * (a - 1.0), np.eye(3) * L


_BALL = None


def _cluster(rng, n):
    """n atoms of a spherical cluster at the same density, no cell."""
    global _BALL
    a = 1.85
    if _BALL is None:
        g = np.array(list(itertools.product(range(-6, 7), repeat=3)), np.float64) * a
        r = np.linalg.norm(g, axis=1)
        k = np.argsort(r, kind="stable")
        _BALL = g[k], r[k]
    R = (3 * n / (4 * math.pi * 0.08)) ** (1 / 3)
    m = max(n, int(np.searchsorted(_BALL[1], R)))
    return _BALL[0][:m][rng.permutation(m)[:n]] + rng.uniform(-0.5, 0.5, (n, 3)) * (a - 1.0)


def _batch(case, rng, part):
    """Structures of 8 to 256 atoms (log-uniform), alternately periodic cubes
    and clusters, each of 1 to 5 of the table's elements.  The sizes belong to
    the case, the structures to the seed."""
    draw = np.random.default_rng([17, part, case["structures"]])
    sizes = np.clip(np.floor(np.exp(draw.uniform(math.log(8), math.log(257), case["structures"]))), 8, 256).astype(np.int64)
    pos, cells, pbc, sp = [], [], [], []
    for s, n in enumerate(sizes.tolist()):
        if s % 2 == 0:
            p, cell = _cube(rng, n)
        else:
            p, cell = _cluster(rng, n), np.zeros((3, 3))
        k = int(rng.integers(1, min(5, case["n_el"]) + 1))
        els = rng.permutation(case["n_el"])[:k]
        pos.append(p)
        cells.append(cell)
        pbc.append([s % 2 == 0] * 3)
        sp.append(els[rng.integers(0, k, n)])
    return (np.concatenate(pos), np.concatenate(sp).astype(np.int32), np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64),
            np.stack(cells), np.array(pbc, np.uint8))


def _structures(case, seed, part=0):
    """(positions, species, atom_off, cells, pbc) as numpy arrays.  The rows
    of a dense Jacobian are counted by the neighbor pairs: there the geometry
    belongs to the case, and the seed gives the species and the place."""
    rng = geo = np.random.default_rng([int(seed), part])
    if case["call"] == "jacobian":
        geo = np.random.default_rng([23, part])
    if case["system"] == "batch":
        pos, sp, off, cells, pbc = _batch(case, geo, part)
        if geo is not rng:
            pos, sp = pos + rng.uniform(0.0, 1.0, 3), rng.permutation(sp)
        return pos, sp, off, cells, pbc
    if case["system"] == "box":
        n = case["atoms"]
        pos, cell = _cube(geo, n)
        if n == 64:  # the repository's box: 64 atoms in a 10 A cube
            pos, cell = pos * (10.0 / cell[0, 0]), np.eye(3) * 10.0
    else:
        pos, cell = synth.fcc_supercell(geo, case["a"], (case["nx"], case["ny"], case["nz"]), case["jitter"], case["vacuum"])
        pos = np.delete(pos, geo.permutation(len(pos))[: case["vacancies"]], axis=0)
    pos = pos + rng.uniform(0.0, 1.0, 3)  # where the structure lies in its cell
    sp = rng.integers(0, case["n_el"], len(pos)).astype(np.int32)
    return np.ascontiguousarray(pos), sp, np.array([0, len(pos)], np.int64), cell.reshape(1, 3, 3), np.ones((1, 3), np.uint8)


def _points(case, seed, atom_off, cells, pbc):
    """Reference points, shared out over the structures: uniform in a
    structure's cell, or around the cluster's centre."""
    rng = np.random.default_rng([int(seed), 77])
    S, n = len(cells), case["points"]
    off = (np.arange(S + 1) * n) // S
    pts = np.empty((n, 3))
    for s in range(S):
        k = int(off[s + 1] - off[s])
        if pbc[s].any():
            pts[off[s]:off[s + 1]] = rng.uniform(0, 1, (k, 3)) @ cells[s]
        else:
            R = (3 * int(atom_off[s + 1] - atom_off[s]) / (4 * math.pi * 0.08)) ** (1 / 3)
            pts[off[s]:off[s + 1]] = rng.uniform(-1, 1, (k, 3)) * R
    return pts, off.astype(np.int64)


def _n_features(case):
    return int(case["density"]) + (case["lmax"] + 1) * case["n_sigma"]


def _upstream(case, n, seed, device):
    g = torch.Generator(device="cpu" if device == "cpu" else device)
    g.manual_seed(int(seed) * 2 + 1)
    return torch.randn((n, _n_features(case)), generator=g, device=device, dtype=torch.float32)


def prepare(case, seed):
    n_gauss, coef, expo = _table(case)
    F = GMPFeaturizer(_orders(case), _sigmas(case), case["cutoff"], n_gauss, coef, expo)
    state = dict(call=case["call"], F=F, batches=[])
    for part in range(case.get("minibatches", 1)):
        pos, sp, off, cells, pbc = _structures(case, seed, part)
        state["batches"].append((torch.from_numpy(pos).cuda(), torch.from_numpy(sp).cuda(), off, cells, pbc))
    if case["call"] in ("vjp", "virial"):
        state["grad"] = _upstream(case, len(pos), seed, "cuda")
    if case["call"] == "points":
        pts, poff = _points(case, seed, off, cells, pbc)
        state["points"] = (torch.from_numpy(pts).cuda(), poff)
    if case.get("tuned"):
        F.tune(*state["batches"][0], cache=False)
    return state


def run(state):
    F, call, b = state["F"], state["call"], state["batches"]
    if call == "screen":
        return [F.featurize(*x) for x in b]
    if call == "features":
        return F.featurize(*b[0])
    if call == "vjp":
        return F.featurize_vjp(*b[0], state["grad"])
    if call == "virial":  # the stress joins a loss in the features' precision
        feat, grad, vir = F.featurize_vjp_virial(*b[0], state["grad"])
        return feat, grad, vir.float()
    if call == "points":
        return F.featurize_points(*b[0], *state["points"])
    return F.featurize_grad(*b[0])


# --------------------------------------------------------------------- work
def _sizes(case):
    """(atoms, structures, centers, neighbor pairs) of a case, from its
    densities (clusters: the average over the sphere's volume)."""
    rc = case["cutoff"]
    ball = 4 / 3 * math.pi * rc ** 3
    if case["system"] == "batch":
        n = 72.0  # mean of a log-uniform size in 8..256
        S = case["structures"] * case.get("minibatches", 1)
        R = (3 * n / (4 * math.pi * 0.08)) ** (1 / 3)
        inside = 1 - 9 * rc / (16 * R) + (rc / R) ** 3 / 32 if rc < 2 * R else (R / rc) ** 3
        centers, per = n * S, 1 + 0.08 * ball * (0.5 + 0.5 * inside)
        atoms = centers
    else:
        S = 1
        atoms = case["atoms"] if case["system"] == "box" else 4 * case["nx"] * case["ny"] * case["nz"] - case["vacancies"]
        rho = (0.064 if case["atoms"] == 64 else 0.08) if case["system"] == "box" else 4 / case["a"] ** 3
        centers, per = atoms, 1 + rho * ball
    if case["call"] == "points":
        centers = case["points"]
    return atoms, S, centers, centers * per


def work(case):
    """Positions, species and upstream gradients in, features and derivatives
    out; per pair the radial factors (an exponential per sigma and Gaussian,
    a multiply-add per order more), the harmonics and the sums over them, and
    for gradients the two sums with the adjoints."""
    atoms, S, centers, pairs = _sizes(case)
    F, L, ns, K = _n_features(case), case["lmax"], case["n_sigma"], case["n_gauss"]
    ind = (L + 1) ** 2
    io = atoms * 28.0 + S * 72.0 + centers * 4.0 * F
    fma = ns * K * (2 + L) + ns * ind + 4 * ind
    if case["call"] == "points":
        io += centers * 24.0
    if case["call"] in ("vjp", "virial"):
        io += centers * 4.0 * F + atoms * 12.0
        fma += ns * K + 2 * ns * ind + 10 * ind
    if case["call"] == "jacobian":
        io += pairs * (12.0 * F + 4.0)
        fma += ns * K + 4 * ns * ind
    return {"bytes": io, "flops": 2.0 * fma * pairs}


# -------------------------------------------------------------------- exact
def _harmonics(L):
    """Per order: exponents of its monomials, the coefficients of S_abc in
    them, and the weights l!/(a!b!c!).  S_abc = (-1)^l r^(2l+1) d^abc (1/r),
    raised by S_(+v) = (2l+1) v S - r^2 dS/dv."""
    polys = {(0, 0, 0): {(0, 0, 0): 1.0}}
    out = []
    for l in range(L + 1):
        comps = [(a, b, l - a - b) for a in range(l + 1) for b in range(l - a + 1)]
        for c in comps:
            if c in polys:
                continue
            v = next(k for k in range(3) if c[k])
            low = polys[tuple(c[k] - (k == v) for k in range(3))]
            p = {}
            for m, x in low.items():
                up = tuple(m[k] + (k == v) for k in range(3))
                p[up] = p.get(up, 0.0) + (2 * l - 1) * x
                if m[v]:
                    dn = [m[k] - (k == v) for k in range(3)]
                    for w in range(3):
                        q = tuple(dn[k] + 2 * (k == w) for k in range(3))
                        p[q] = p.get(q, 0.0) - m[v] * x
            polys[c] = p
        C = np.array([[polys[c].get(m, 0.0) for m in comps] for c in comps])
        w = np.array([math.factorial(l) / math.prod(math.factorial(k) for k in c) for c in comps])
        out.append((comps, C, w))
    return out


def _pairs(x, centers, ids, cell, pbc, rc):
    """Blocks (center, atom, displacement) of one structure: every atom image
    within rc of the centers, 64-bit.  ids: the centers' numbers."""
    dev = x.device
    ghosts, owner = x, torch.arange(len(x), device=dev)
    base = torch.zeros_like(x)
    lo, hi = centers.min(0).values - rc - 1e-6, centers.max(0).values + rc + 1e-6
    if pbc.any():
        inv = np.linalg.inv(cell)
        u = x.cpu().numpy() @ inv
        uc = centers.cpu().numpy() @ inv
        span = np.maximum(uc.max(0) - u.min(0), u.max(0) - uc.min(0))
        M = [int(math.ceil(rc * np.linalg.norm(inv[:, k]) + span[k])) if pbc[k] else 0 for k in range(3)]
        A = torch.as_tensor(cell, dtype=torch.float64, device=dev)
        g, o, b = [], [], []
        for n in itertools.product(*(range(-m, m + 1) for m in M)):
            sh = (n[0] * A[0] + n[1] * A[1]) + n[2] * A[2]
            p = x + sh
            if len(x) > 512:
                keep = ((p >= lo) & (p <= hi)).all(1).nonzero()[:, 0]
            else:
                keep = owner
            g.append(p[keep])
            o.append(owner[keep])
            b.append(sh.expand(len(keep), 3))
        ghosts, owner, base = torch.cat(g), torch.cat(o), torch.cat(b)
    if len(centers) * len(ghosts) <= 40_000_000:
        blocks = [torch.arange(len(centers), device=dev)]
    else:
        edge = 2 * rc
        key = ((centers - lo) / edge).floor().long()
        key = (key[:, 0] * 4096 + key[:, 1]) * 4096 + key[:, 2]
        order = torch.argsort(key)
        cuts = torch.unique_consecutive(key[order], return_counts=True)[1].tolist()
        blocks = torch.split(order, cuts)
    for blk in blocks:
        c = centers[blk]
        if len(blocks) > 1:
            near = ((ghosts >= c.min(0).values - rc - 1e-6) & (ghosts <= c.max(0).values + rc + 1e-6)).all(1).nonzero()[:, 0]
        else:
            near = torch.arange(len(ghosts), device=dev)
        d = (x[owner[near]][None] - c[:, None]) + base[near][None]
        i, j = ((d * d).sum(-1) < rc * rc).nonzero(as_tuple=True)
        yield ids[blk[i]], owner[near[j]], d[i, j]


class _Exact:
    """Features (and derivatives) of chunks of pairs in 64-bit torch."""

    def __init__(self, case, device):
        self.case, self.dev, self.harm = case, device, _harmonics(case["lmax"])
        n_gauss, coef, expo = _table(case)
        K = case["n_gauss"]
        t = lambda v: torch.as_tensor(np.asarray(v), dtype=torch.float64, device=device)  # noqa: E731
        a, c = t(expo).reshape(-1, 1, K), t(coef).reshape(-1, 1, K)
        sig = t(_sigmas(case)).reshape(1, -1, 1)
        beta = 1 / (2 * sig * sig)
        g = a + beta
        self.rate = a * beta / g
        A0 = c * (2 * math.pi * sig * sig) ** -1.5 * (math.pi / g) ** 1.5
        self.amp = torch.stack([A0 * (a / g) ** l for l in range(case["lmax"] + 1)], 1)  # [el, l, s, K]
        self.dens_a, self.dens_c = a.reshape(-1, K), c.reshape(-1, K)
        self.coef = [t(C) for _, C, _ in self.harm]
        self.weight = [t(w) for _, _, w in self.harm]

    def monomials(self, d):
        pw = [[torch.ones_like(d[:, 0])] for _ in range(3)]
        for k in range(3):
            for _ in range(self.case["lmax"]):
                pw[k].append(pw[k][-1] * d[:, k])
        return [torch.stack([pw[0][a] * pw[1][b] * pw[2][c] for a, b, c in comps], 1) for comps, _, _ in self.harm]

    def radial(self, e, d):
        """[P, l, s] radial factors, d/dr2 of them, and the density terms."""
        r2 = (d * d).sum(-1)
        R = d.new_empty(len(d), self.case["lmax"] + 1, self.case["n_sigma"])
        parts, back, dens = [], [], []
        for el in range(self.case["n_el"]):
            at = (e == el).nonzero()[:, 0]
            E = torch.exp(-self.rate[el][None] * r2[at][:, None, None])
            parts.append(torch.einsum("psk,lsk->pls", E, self.amp[el]))
            dens.append((self.dens_c[el] * torch.exp(-self.dens_a[el] * r2[at][:, None])).sum(-1))
            back.append(at)
        inv = torch.argsort(torch.cat(back))
        return torch.cat(parts)[inv], torch.cat(dens)[inv]

    def features(self, n, i, e, d):
        """[n, F] features of the centers 0 .. n-1, and their moments."""
        R, rho = self.radial(e, d)
        out, mus = [], []
        if self.case["density"]:
            out.append(torch.zeros(n, 1, dtype=torch.float64, device=self.dev).index_add(0, i, rho[:, None]))
        for l, mono in enumerate(self.monomials(d)):
            S = mono @ self.coef[l].T
            mu = torch.zeros(n, R.shape[2], S.shape[1], dtype=torch.float64, device=self.dev).index_add(
                0, i, R[:, l, :, None] * S[:, None, :])
            mus.append(mu)
            out.append((mu * mu) @ self.weight[l])
        return torch.cat(out, 1), mus

    def pair_gradients(self, i, e, d, mus):
        """[P, F, 3]: d f(center) / d(displacement) of each pair."""
        r2 = (d * d).sum(-1)
        res = d.new_zeros(len(d), _n_features(self.case), 3)
        at, ns = 0, self.case["n_sigma"]
        if self.case["density"]:
            a, c = self.dens_a[e], self.dens_c[e]
            res[:, 0] = (-2 * a * c * torch.exp(-a * r2[:, None])).sum(-1)[:, None] * d
            at = 1
        E = torch.exp(-self.rate[e] * r2[:, None, None])
        mono = self.monomials(d)
        for l, (comps, C, _) in enumerate(self.harm):
            R = (self.amp[e, l] * E).sum(-1)
            dR = (-self.rate[e] * self.amp[e, l] * E).sum(-1)
            lam = (2 * self.weight[l] * mus[l])[i]  # [P, s, c]
            P = (lam * (mono[l] @ self.coef[l].T)[:, None]).sum(-1)
            for v in range(3):
                g = 2 * d[:, v, None] * dR * P
                if l:
                    low = self.harm[l - 1][0]
                    D = np.zeros((len(comps), len(low)))  # monomial -> its derivative's monomial
                    for m, q in enumerate(comps):
                        if q[v]:
                            D[m, low.index(tuple(q[k] - (k == v) for k in range(3)))] = q[v]
                    dS = mono[l - 1] @ torch.as_tensor(C @ D, device=self.dev).T
                    g = g + R * (lam * dS[:, None]).sum(-1)
                res[:, at + l * ns:at + (l + 1) * ns, v] = g
        return res


def _pass_exact(case, seed, part, device, chunk):
    pos, sp, off, cells, pbc = _structures(case, seed, part)
    x = torch.from_numpy(pos).to(device)
    e_all = torch.from_numpy(sp).long().to(device)
    call, N, F = case["call"], len(pos), _n_features(case)
    if call == "points":
        pts, coff = _points(case, seed, off, cells, pbc)
        centers = torch.from_numpy(pts).to(device)
    else:
        centers, coff = x, off
    X = _Exact(case, device)
    feat = torch.zeros(len(centers), F, dtype=torch.float64, device=device)
    deriv = call in ("vjp", "virial")
    grad = torch.zeros(N, 3, dtype=torch.float64, device=device)
    vir = torch.zeros(len(cells), 3, 3, dtype=torch.float64, device=device)
    up = _upstream(case, N, seed, device).double() if deriv else None
    rows = []

    def flush(held):
        i, j, d, s = (torch.cat(v) for v in zip(*held))
        who, local = torch.unique(i, return_inverse=True)
        d.requires_grad_(deriv)
        f, mus = X.features(len(who), local, e_all[j], d)
        feat[who] = f.detach()
        if deriv:
            (gd,) = torch.autograd.grad((f * up[who]).sum(), d)
            grad.index_add_(0, j, gd)
            grad.index_add_(0, i, -gd)
            vir.index_add_(0, s, gd[:, :, None] * d.detach()[:, None, :])
        if call == "jacobian":  # one row per center and neighbor atom, the own row minus the others' sum
            g = X.pair_gradients(local, e_all[j], d, mus)
            key, at = torch.unique(i * N + j, return_inverse=True)
            J = torch.zeros(len(key), F, 3, dtype=torch.float64, device=device).index_add(0, at, g)
            own = key // N == key % N
            J[own] = 0
            J[own] = -torch.zeros(len(who), F, 3, dtype=torch.float64, device=device).index_add(
                0, torch.searchsorted(who, key // N), J)
            rows.append((key, J))

    held, count = [], 0
    for s in range(len(cells)):
        a, b = int(off[s]), int(off[s + 1])
        ca, cb = int(coff[s]), int(coff[s + 1])
        if b == a or cb == ca:
            continue
        ids = torch.arange(ca, cb, device=device)
        for i, j, d in _pairs(x[a:b], centers[ca:cb], ids, cells[s], pbc[s], case["cutoff"]):
            held.append((i, j + a, d, torch.full_like(i, s)))
            count += len(i)
            if count >= chunk:
                flush(held)
                held, count = [], 0
    if count:
        flush(held)
    if call == "vjp":
        return feat, grad
    if call == "virial":
        return feat, grad, vir
    if call == "jacobian":
        key = torch.cat([k for k, _ in rows])
        return feat, None, None, torch.cat([J for _, J in rows])[torch.argsort(key)]
    return feat


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    chunk = 400_000 if case["call"] != "jacobian" else 100_000
    parts = [_pass_exact(case, seed, p, device, chunk) for p in range(case.get("minibatches", 1))]
    return parts if case["call"] == "screen" else parts[0]
