"""The work that users of the GW sweep have it do, as timed cases.

Every case goes through the public binding (``paper_1911_05633_gb300.gw``): whole sweeps,
the rows of a sweep one by one, the batch of uneven systems, the W solve over the sizes a
product basis gives it, the Dyson step with its chemical potential, and the band and
spectral calls.  The cells are the repository's own: the two-atom simple cubic cell, the
diamond-like supercells and the layered perovskite-like cell, with the grids, meshes,
cutoffs and basis sizes of its configurations and their neighbours (odd node counts, bases
that are no multiple of a tile, meshes without quarter-turn phases).

``listed`` gives the cases, ``draw`` one more of the same ranges, ``prepare`` the inputs
and the plan a program holds before the call, ``run`` one pass, ``work`` what a pass cannot
do without, ``exact`` the result in 64-bit arithmetic from torch and numpy alone.
"""
import math

import numpy as np
import torch

from paper_1911_05633_gb300 import gw

DEV = "cuda"
CD = torch.complex128
FCC = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
DIAMOND = np.vstack([FCC, FCC + 0.25])
# K2NiF4-type layered cell: transition-metal sites, anions, A-site cations
LAYERED = np.array([[0, 0, 0], [.5, .5, .5], [.5, 0, 0], [0, .5, 0], [.5, 0, .5], [0, .5, .5], [0, 0, .182],
                    [0, 0, .818], [.5, .5, .318], [.5, .5, .682], [0, 0, .362], [0, 0, .638], [.5, .5, .138],
                    [.5, .5, .862]])
LAYERED_SPECIES = [0, 0, 2, 2, 2, 2, 2, 2, 2, 2, 1, 1, 1, 1]


def listed():
    d8 = dict(cell="diamond-1x1x1", mesh="4x4x4", cutoff=12.0, n=9, K=48, nt=48, beta=1000.0)
    d16 = dict(cell="diamond-2x1x1", mesh="2x2x2", cutoff=12.0, n=9, K=64, nt=64, beta=1000.0)
    return [
        # the smallest system a user runs, one whole FP64 sweep: launches and latency
        dict(name="sweep-2atoms-fp64", kind="sweep", cell="cubic-1x1x1", mesh="2x2x2", cutoff=0.0, n=4, K=8, nt=24,
             beta=50.0, precision="fp64"),
        # the headline workload: the P and Sigma rows of the 72-atom supercell, mixed precision
        dict(name="rows-72atoms-mixed", kind="rows", cell="diamond-3x3x1", mesh="2x2x2", cutoff=12.0, n=9, K=64, nt=64,
             beta=1000.0, precision="mixed"),
        # the FP64 polarizability of the 8-atom silicon-like cell
        dict(name="p-8atoms-fp64", kind="p", precision="fp64", **d8),
        # the FP64 self-energy and exchange with the three product-basis levels of distance
        dict(name="sigma-8atoms-levels-fp64", kind="sigma", precision="fp64", r_b=4.6, K_near=36, K_far=24, **d8),
        # the mixed contractions of uneven systems as one batch (diamond-like cells, one layered oxide)
        dict(name="batch-5systems-mixed", kind="batch", n=9, K=48, nt=48, beta=1000.0,
             cells="diamond-1x1x1/3x3x3/10,diamond-2x1x1/2x2x2/12,diamond-1x1x1/4x4x4/12,diamond-3x1x1/2x2x2/10,"
                   "layered-1x1x1/2x2x2/12"),
        # the tau <-> i omega transforms of one iteration: P, W~ and Sigma
        dict(name="tau-16atoms", kind="tau", **d16),
        # the lattice transforms on a mesh without quarter-turn phases: G, v and Sigma
        dict(name="lattice-16atoms-k3", kind="lattice", cell="diamond-2x1x1", mesh="3x3x3", cutoff=14.0, n=9, K=48,
             nt=48, beta=1000.0),
        # the screened interaction of the 8-atom cell (order 384)
        dict(name="w-order384", kind="w", **d8),
        # the screened interaction of a 16-atom supercell (order 1024)
        dict(name="w-order1024", kind="w", **d16),
        # the screened interaction for a product basis whose order is no multiple of a tile
        dict(name="w-order288", kind="w", cell="diamond-1x1x1", mesh="3x3x3", cutoff=10.0, n=9, K=36, nt=24, beta=200.0),
        # the end of an iteration: the chemical potential of the new Sigma and the Dyson step
        dict(name="dyson-8atoms", kind="dyson", **dict(d8, beta=200.0)),
        # after convergence: quasiparticle bands, the continued Sigma and the spectral function
        dict(name="bands-8atoms", kind="bands", n_real=64, delta=0.05, **dict(d8, beta=200.0)),
    ]


def draw(rng):
    def mesh(most):
        while True:
            m = [rng.randint(1, 4) for _ in range(3)]
            if 2 <= m[0] * m[1] * m[2] <= most:
                return "%dx%dx%d" % tuple(m)

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["sweep", "rows", "p", "sigma", "batch", "tau", "lattice", "w", "w", "dyson", "bands"])
    c = dict(kind=kind, cell="diamond-%s" % rng.choice(["1x1x1", "2x1x1", "3x1x1", "2x2x1"]), mesh=mesh(27),
             cutoff=rng.choice([7.5, 9.0, 10.0, 12.0, 14.0]), n=rng.choice([4, 5, 8, 9, 9, 9]), K=log(8, 64),
             nt=rng.randint(15, 64), beta=float(log(50, 1000)))
    if kind == "sweep":
        c.update(cell=rng.choice(["cubic-1x1x1", "cubic-2x1x1", "cubic-2x2x1"]), cutoff=0.0, n=rng.randint(1, 5),
                 K=log(4, 24), nt=rng.randint(9, 32), beta=float(log(10, 100)), mesh=mesh(12), precision="fp64")
    elif kind in ("rows", "p", "sigma"):
        c["precision"] = rng.choice(["fp64", "mixed"]) if kind != "rows" else "mixed"
        if kind != "rows" and rng.random() < 0.3:
            c.update(r_b=4.6, K_near=max(1, c["K"] * 3 // 4), K_far=max(1, c["K"] // 2))
        if kind != "rows" and rng.random() < 0.2:
            c.update(cell="layered-1x1x1", mesh=mesh(8), nt=rng.randint(15, 48), cutoff=10.0)
    elif kind == "batch":
        pool = ["diamond-1x1x1/3x3x3/10", "diamond-1x1x1/2x3x2/12", "diamond-2x1x1/2x2x2/12", "diamond-2x1x1/3x2x1/10",
                "diamond-3x1x1/2x2x2/10", "layered-1x1x1/2x2x2/10", "cubic-1x1x1/2x2x2/0", "cubic-2x1x1/3x2x2/12"]
        c = dict(kind="batch", n=c["n"], K=log(16, 64), nt=rng.randint(15, 48), beta=c["beta"],
                 cells=",".join(rng.sample(pool, rng.randint(2, 5))))
    elif kind == "w":
        cell, atoms = rng.choice([("cubic-1x1x1", 2), ("diamond-1x1x1", 8), ("diamond-1x1x1", 8), ("diamond-2x1x1", 16)])
        order = log(24, 384) if atoms < 16 else rng.choice([512, 640, 768, 896, 1024, 16 * rng.randint(25, 47)])
        c.update(cell=cell, K=max(4, min(96, order // atoms)), n=9 if atoms > 2 else 5, nt=rng.randint(15, 40),
                 mesh=mesh(27 if atoms < 16 else 8 if order % 128 == 0 else 4))
    elif kind in ("dyson", "bands"):
        c.update(cell=rng.choice(["cubic-1x1x1", "cubic-2x1x1", "diamond-1x1x1"]), n=rng.choice([4, 5, 8, 9]),
                 nt=rng.randint(16, 48), beta=float(log(20, 200)), mesh=mesh(64))
        if kind == "bands":
            c.update(n_real=log(8, 64), delta=0.05)
    return c


# ---- the system of a case ---------------------------------------------------------------

class Cell:
    """Geometry, basis and grids of one system; `seed` sets the product-basis coefficients."""

    def __init__(self, case, seed, text=None, mesh=None, cutoff=None):
        text = text or case["cell"]
        kind, mult = text.split("-")
        m = np.array([int(x) for x in mult.split("x")])
        self.mesh = tuple(int(x) for x in (mesh or case["mesh"]).split("x"))
        self.cutoff = float(case["cutoff"] if cutoff is None else cutoff)
        base, spec, lat = {"cubic": (np.array([[0, 0, 0], [.5, .5, .5]]), [0, 0], [5.0, 5.0, 5.0]),
                           "diamond": (DIAMOND, [0] * 8, [10.26] * 3),
                           "layered": (LAYERED, LAYERED_SPECIES, [7.14, 7.14, 24.85])}[kind]
        self.frac = np.vstack([(base + np.array(s)) / m for s in np.ndindex(*m)])
        self.species = np.tile(np.array(spec, np.int32), int(m.prod()))
        self.lattice = np.diag(np.array(lat) * m)
        self.n_orb, self.n_prod = ([14, 9, 9], [96, 64, 40]) if kind == "layered" else ([case["n"]], [case["K"]])
        self.r_b = float(case.get("r_b", 0.0))
        scale = lambda key: [max(1, k * case[key] // case["K"]) for k in self.n_prod] if self.r_b else list(self.n_prod)  # noqa: E731
        self.n_near, self.n_far = scale("K_near"), scale("K_far")
        self.beta, self.nt = float(case["beta"]), int(case["nt"])
        rng = np.random.default_rng([seed, len(self.frac)])
        self.C = []
        for n, k in zip(self.n_orb, self.n_prod):
            x = rng.standard_normal((k, n, n))
            self.C.append(0.5 * (x + x.transpose(0, 2, 1)) / n)
        t = 0.5 * self.beta * (1.0 - np.cos(np.pi * np.arange(self.nt) / (self.nt - 1)))
        t[0], t[-1] = 0.0, self.beta
        half = self.nt // 2
        t[self.nt - 1 - np.arange(half)] = self.beta - t[:half]
        self.tau = t
        npos = (self.nt + 1) // 2
        idx = list(range(min(max(1, round(0.375 * self.nt)), npos)))
        for g in np.geomspace(max(1, len(idx)), 3 * self.nt, npos - len(idx)) if npos > len(idx) else []:
            idx.append(max(int(round(g)), idx[-1] + 1))
        idx = np.array(idx)
        self.om = np.sort(np.concatenate([idx, -idx - 1]))
        self.nu = np.sort(np.concatenate([[0], idx + 1, -(idx + 1)]))
        self.nat, self.nk = len(self.frac), int(np.prod(self.mesh))
        self.oo = np.concatenate([[0], np.cumsum([self.n_orb[s] for s in self.species])])
        self.po = np.concatenate([[0], np.cumsum([self.n_prod[s] for s in self.species])])
        self.N, self.NP = int(self.oo[-1]), int(self.po[-1])

    def plan(self, **kw):
        if self.r_b:
            kw.update(r_b=self.r_b, n_prod_far=self.n_far, n_prod_near=self.n_near)
        return gw.Plan(self.lattice, self.frac, self.species, self.n_orb, self.n_prod, self.C, self.mesh, self.beta,
                       self.tau, self.om, self.nu, self.cutoff, **kw)

    def distances(self):
        """Minimum-image distance of every (a, b, class), [nat][nat][nk]."""
        cls = np.array(list(np.ndindex(*self.mesh)))
        d0 = self.frac[None, :] - self.frac[:, None]
        best = np.full((self.nat, self.nat, self.nk), np.inf)
        for s in np.ndindex(3, 3, 3):
            R = cls + (np.array(s) - 1) * np.array(self.mesh)
            x = (d0[:, :, None, :] + R[None, None]) @ self.lattice
            best = np.minimum(best, np.sqrt((x * x).sum(-1)))
        return best

    def entries(self):
        """Groups of pair entries of one block shape, in the order of (a, b, class): a list of
        (a, b, class, place in the list), the block dims per kind, and the offsets."""
        if not hasattr(self, "_ent"):
            d = self.distances()
            keep = np.ones_like(d, bool) if self.cutoff <= 0 else d <= self.cutoff
            a, b, c = np.nonzero(keep)
            d = d[a, b, c]
            tier = np.where((a == b) & (d < 1e-6), 0, np.where((self.r_b > 0) & (d * d > self.r_b ** 2 + 1e-9), 2, 1))
            sizes = np.array([self.n_prod, self.n_near, self.n_far])
            dims = {"orb": (np.array(self.n_orb)[self.species[a]], np.array(self.n_orb)[self.species[b]]),
                    "pb": (sizes[tier, self.species[a]], sizes[tier, self.species[b]])}
            off = {k: np.concatenate([[0], np.cumsum(r * q)]) for k, (r, q) in dims.items()}
            key = ((dims["pb"][0] * 1000 + dims["pb"][1]) * 100 + self.species[a]) * 100 + self.species[b]
            groups = [np.nonzero(key == x)[0] for x in np.unique(key)]
            self._ent = (a, b, c, groups, dims, off)
        return self._ent

    def length(self, kind):
        return int(self.entries()[5][kind][-1])


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + salt)
    return g


def _randc(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV, dtype=torch.float64))


def hamiltonian(cell, seed, split):
    """Tight-binding H(k): onsite levels in [-0.5, 0.5] Ha moved apart by `split`, hoppings of
    magnitude 0.1 exp(-d/2) with random phases; and the half-filling chemical potential."""
    g = _gen(seed, 1)
    nmax, nat = max(cell.n_orb), cell.nat
    shifts = [math.ceil(10.0 / cell.lattice[i, i]) for i in range(3)]
    R = np.array([np.array(s) - shifts for s in np.ndindex(*[2 * s + 1 for s in shifts])])
    x = (cell.frac[None, :, None] - cell.frac[:, None, None] + R[None, None]) @ cell.lattice
    d = np.sqrt((x * x).sum(-1))
    a, b, r = np.nonzero((d <= 10.0) & (d > 1e-6))
    mag = torch.from_numpy(0.1 * np.exp(-d[a, b, r] / 2)).to(DEV)
    ang = torch.rand(len(a), nmax * nmax, generator=g, device=DEV, dtype=torch.float64) * (2 * math.pi)
    blk = torch.polar(mag[:, None].expand_as(ang).contiguous(), ang)
    kf = np.array(list(np.ndindex(*cell.mesh))) / np.array(cell.mesh)
    ph = np.exp(2j * np.pi * (kf @ R[r].T))
    pair, first = np.unique(a * nat + b, return_index=True)  # the hoppings come sorted by (a, b)
    H = np.zeros((cell.nk, nat * nat, nmax * nmax), np.complex128)
    H[:, pair] = np.add.reduceat(ph[:, :, None] * blk.cpu().numpy()[None], first, axis=1)
    H = torch.from_numpy(H).to(DEV).view(cell.nk, nat, nat, nmax, nmax).transpose(2, 3).reshape(cell.nk, nat * nmax, nat * nmax)
    keep = torch.from_numpy(np.concatenate([at * nmax + np.arange(cell.n_orb[s]) for at, s in enumerate(cell.species)])).to(DEV)
    H = H[:, keep][:, :, keep]
    lev = torch.rand(cell.N, generator=g, device=DEV, dtype=torch.float64) - 0.5
    lev = lev + split * torch.where(lev < lev.median(), -0.5, 0.5)
    H = 0.5 * (H + H.mH) + torch.diag(lev).to(CD)
    e, U = torch.linalg.eigh(H)
    s = e.reshape(-1).sort().values
    h = cell.nk * cell.N // 2
    return H.contiguous(), e, U, float(0.5 * (s[max(0, h - 1)] + s[h]))


def _g0(xi, t, beta):
    """-e^{-xi t} / (1 + e^{-beta xi}), without overflow."""
    return -1.0 / (torch.exp(torch.clamp(xi * t, -700, 700)) + torch.exp(torch.clamp(xi * (t - beta), -700, 700)))


def green(cell, seed):
    """G(k, tau) [nk][nt][N][N] of the tight-binding cell."""
    _, e, U, mu = hamiltonian(cell, seed, 0.6)
    t = torch.from_numpy(cell.tau).to(DEV)
    G = torch.empty(cell.nk, cell.nt, cell.N, cell.N, dtype=CD, device=DEV)
    for k in range(cell.nk):
        torch.matmul(U[k] * _g0((e[k] - mu)[None, :], t[:, None], cell.beta)[:, None, :], U[k].mH, out=G[k])
    return G


def to_entries(cell, kind, F):
    """F(R) of dense F(k) [nk][S][N][N] in the entry layout, by torch's FFT over the mesh."""
    S, N = F.shape[1], F.shape[2]
    Fc = torch.fft.fftn(F.view(*cell.mesh, S, N, N), dim=(0, 1, 2), norm="forward").view(cell.nk, S, N, N)
    a, b, c, groups, dims, off = cell.entries()
    o = cell.po if kind == "pb" else cell.oo
    blocks = []
    for g in groups:
        r, q = int(dims[kind][0][g[0]]), int(dims[kind][1][g[0]])
        cl, ri, ci = (torch.from_numpy(x).to(DEV) for x in (c[g], o[a[g]][:, None] + np.arange(r), o[b[g]][:, None] + np.arange(q)))
        blocks.append(Fc[cl[:, None, None, None], torch.arange(S, device=DEV)[None, :, None, None],
                         ri[:, None, :, None], ci[:, None, None, :]])
    return join(cell, kind, S, blocks)


def to_dense(cell, kind, S, flat):
    """F(k) = sum over the kept entries of e^{ik.R} F(R), dense [nk][S][N][N]."""
    a, b, c, groups, dims, _ = cell.entries()
    o, N = (cell.po, cell.NP) if kind == "pb" else (cell.oo, cell.N)
    Fc = torch.zeros(cell.nk, S, N, N, dtype=CD, device=DEV)
    for g, blk in zip(groups, split(cell, kind, S, flat)):
        cl, ri, ci = (torch.from_numpy(x).to(DEV) for x in (c[g], o[a[g]][:, None] + np.arange(blk.shape[2]),
                                                            o[b[g]][:, None] + np.arange(blk.shape[3])))
        Fc[cl[:, None, None, None], torch.arange(S, device=DEV)[None, :, None, None],
           ri[:, None, :, None], ci[:, None, None, :]] = blk
    return torch.fft.ifftn(Fc.view(*cell.mesh, S, N, N), dim=(0, 1, 2), norm="forward").reshape(cell.nk, S, N, N)


def _places(cell, kind, S, g):
    dims, off = cell.entries()[4:]
    blk = int(dims[kind][0][g[0]] * dims[kind][1][g[0]])
    return (torch.from_numpy(off[kind][g]).to(DEV)[:, None] * S + torch.arange(S * blk, device=DEV)[None, :])


def join(cell, kind, S, blocks):
    """Blocks per group -> the flat entry layout."""
    groups = cell.entries()[3]
    if len(groups) == 1:
        return blocks[0].reshape(-1).contiguous()
    out = torch.empty(S * cell.length(kind), dtype=blocks[0].dtype, device=DEV)
    for g, blk in zip(groups, blocks):
        out[_places(cell, kind, S, g)] = blk.reshape(len(g), -1)
    return out


def split(cell, kind, S, flat):
    """The flat entry layout -> blocks [entries][S][rows][cols] per group."""
    groups, dims = cell.entries()[3:5]
    if len(groups) == 1:
        g = groups[0]
        return [flat.view(len(g), S, int(dims[kind][0][g[0]]), int(dims[kind][1][g[0]]))]
    return [flat[_places(cell, kind, S, g)].view(len(g), S, int(dims[kind][0][g[0]]), int(dims[kind][1][g[0]])) for g in groups]


def spread(cell, kind, g, f):
    """Entry-layout values out[e][s][element] = sum_p amplitude[e][element][p] f[p][s]: seeded
    amplitudes falling off with the entry's distance, the time or frequency shape from f."""
    dist = cell.distances()
    a, b, c, groups, dims, _ = cell.entries()
    blocks = []
    for gr in groups:
        r, q = int(dims[kind][0][gr[0]]), int(dims[kind][1][gr[0]])
        amp = torch.randn(len(gr), f.shape[0], r * q, generator=g, device=DEV, dtype=torch.float64)
        amp /= (1.0 + torch.from_numpy(dist[a[gr], b[gr], c[gr]]).to(DEV))[:, None, None]
        blocks.append(torch.matmul(f.t()[None], amp.to(f.dtype)).view(len(gr), f.shape[1], r, q))
        del amp
    return join(cell, kind, f.shape[1], blocks)


def boson_tau(cell):
    """Shapes in tau of a bosonic function with F(beta - tau) = F(tau)*: even real, odd imaginary."""
    t = cell.tau
    f = [np.exp(-w * t) + np.exp(-w * (cell.beta - t)) for w in (0.05, 0.5, 2.0)]
    f += [1j * (np.exp(-w * t) - np.exp(-w * (cell.beta - t))) for w in (0.1, 1.0)]
    return torch.from_numpy(np.array(f, np.complex128)).to(DEV)


def boson_nu(cell):
    """Shapes over the bosonic frequencies of a real W~(R, i nu): even and odd parts."""
    v = 2 * np.pi * cell.nu / cell.beta
    f = [2 * w / (v * v + w * w) for w in (0.1, 0.5, 2.0)] + [v / (v * v + w * w) for w in (0.3, 1.0)]
    return torch.from_numpy(np.array(f, np.complex128)).to(DEV)


def fermion_tau(cell):
    """Shapes in tau of a fermionic function: decays from either end, real and imaginary."""
    t = cell.tau
    f = [z * np.exp(-w * t) for z, w in ((1, 0.05), (1j, 0.6))] + [z * np.exp(-w * (cell.beta - t)) for z, w in ((1, 0.2), (1j, 1.0))]
    return torch.from_numpy(np.array(f, np.complex128)).to(DEV)


def coulomb_q(cell, seed):
    """v(q) [nk][NP][NP]: a seeded positive block over 1 + d, its lattice sum, at least 0.05 I."""
    kmax = max(cell.n_prod)
    A = np.random.default_rng([seed, 7]).standard_normal((kmax, kmax))
    X = torch.from_numpy(A @ A.T / kmax + 0.1 * np.eye(kmax)).to(DEV).to(CD)
    cls = np.array(list(np.ndindex(*cell.mesh)))
    ph = np.exp(2j * np.pi * (cls / np.array(cell.mesh)) @ cls.T)
    f = torch.from_numpy(np.einsum("qc,abc->qab", ph, 1.0 / (1.0 + cell.distances()))).to(DEV)
    idx = np.concatenate([np.arange(cell.n_prod[s]) for s in cell.species])
    at = np.concatenate([[i] * cell.n_prod[s] for i, s in enumerate(cell.species)])
    v = f[:, at][:, :, at] * X[idx][:, idx]
    v = 0.5 * (v + v.mH)
    low = float(torch.linalg.eigvalsh(v).min())
    return v + max(0.0, 0.05 - low) * torch.eye(cell.NP, device=DEV, dtype=torch.float64)


def self_energy_k(cell, seed, w):
    """Sigma_c(k, w) [nk][len(w)][N][N] from a few Hermitian positive residues at real levels,
    and a Hermitian Sigma_x(k), for complex frequencies w."""
    g = _gen(seed, 5)
    poles = np.linspace(-1.6, 1.6, 8) + 0.01 * np.random.default_rng([seed, 3]).standard_normal(8)
    B = _randc(g, cell.nk, len(poles), cell.N, cell.N) / cell.N
    res = 0.02 * (B @ B.mH)
    f = torch.from_numpy(1.0 / (np.asarray(w)[:, None] - poles[None, :])).to(DEV)
    S = (f[None] @ res.view(cell.nk, len(poles), -1)).view(cell.nk, len(w), cell.N, cell.N)
    x = _randc(g, cell.nk, cell.N, cell.N)
    return S.contiguous(), (0.05 / math.sqrt(cell.N) * (x + x.mH)).contiguous()


# ---- the 64-bit values ------------------------------------------------------------------

def fourier(cell, stat):
    """T [n_freq][n_tau]: exact Fourier integrals of the polynomial through the tau nodes."""
    x = 2.0 * cell.tau / cell.beta - 1.0
    w = np.array([1.0 / np.prod(2 * (xi - np.delete(x, i))) for i, xi in enumerate(x)])
    a = (2 * cell.om + 1) * np.pi / 2 if stat == "F" else cell.nu * np.pi
    gx, gw_ = np.polynomial.legendre.leggauss(48)
    out = np.empty((len(a), cell.nt), np.complex128)
    for r, ar in enumerate(a):
        e = np.linspace(-1, 1, math.ceil(abs(ar) / 4) + 2)
        h = 0.5 * (e[1:] - e[:-1])
        xg = (0.5 * (e[1:] + e[:-1])[:, None] + h[:, None] * gx).reshape(-1)
        q = w[None] / (xg[:, None] - x[None])
        out[r] = 0.5 * cell.beta * np.exp(1j * ar) * (((h[:, None] * gw_).reshape(-1) * np.exp(1j * ar * xg)) @ (q / q.sum(1, keepdims=True)))
    return out


def along(cell, kind, T, flat):
    """out[e][m] = sum_i T[m][i] in[e][i] in the entry layout."""
    Tt = torch.from_numpy(np.ascontiguousarray(T)).to(DEV)
    out = [torch.matmul(Tt[None], b.reshape(b.shape[0], b.shape[1], -1).to(CD)).view(b.shape[0], T.shape[0], *b.shape[2:])
           for b in split(cell, kind, T.shape[1], flat)]
    return join(cell, kind, T.shape[0], out)


def _chunks(n, per):
    step = max(1, int(per))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _pair_c(cell, g, Ka, Kb):
    a, b = cell.entries()[:2]
    return tuple(torch.from_numpy(cell.C[cell.species[i[g[0]]]][:K]).to(DEV).to(CD) for i, K in ((a, Ka), (b, Kb)))


def polarizability(cell, G_R):
    out = []
    dims, groups = cell.entries()[4], cell.entries()[3]
    for g, G in zip(groups, split(cell, "orb", cell.nt, G_R)):
        Ka, Kb = int(dims["pb"][0][g[0]]), int(dims["pb"][1][g[0]])
        Ca, Cb = _pair_c(cell, g, Ka, Kb)
        na, nb = G.shape[2:]
        P = torch.empty(len(g), cell.nt, Ka, Kb, dtype=CD, device=DEV)
        for i, j in _chunks(len(g), 2e8 / (cell.nt * Ka * max(nb * nb, na * nb))):
            x = torch.einsum("kab,etac->etkbc", Ca, G[i:j])
            y = torch.einsum("etkbc,etbd->etkcd", x, G[i:j].flip(1).conj())
            P[i:j] = -2.0 * torch.matmul(y.reshape(j - i, cell.nt, Ka, -1), Cb.reshape(Kb, -1).t())
        out.append(P)
    return join(cell, "pb", cell.nt, out)


def sigma(cell, G_R, W, S, sign=-1.0):
    out = []
    dims, groups = cell.entries()[4], cell.entries()[3]
    for g, G, w in zip(groups, split(cell, "orb", S, G_R), split(cell, "pb", S, W)):
        Ka, Kb = int(dims["pb"][0][g[0]]), int(dims["pb"][1][g[0]])
        Ca, Cb = _pair_c(cell, g, Ka, Kb)
        na, nb = G.shape[2:]
        Sg = torch.empty(len(g), S, na, nb, dtype=CD, device=DEV)
        for i, j in _chunks(len(g), 2e8 / (S * Ka * max(nb * nb, na * nb))):
            B = torch.matmul(w[i:j].to(CD), Cb.reshape(Kb, -1)).view(j - i, S, Ka, nb, nb)
            h = torch.einsum("klm,etmn->etkln", Ca, G[i:j])
            Sg[i:j] = sign * torch.einsum("etkln,etkpn->etlp", h, B)
        out.append(Sg)
    return join(cell, "orb", S, out)


def last_slice(cell, kind, S, flat):
    return join(cell, kind, 1, [b[:, -1:] for b in split(cell, kind, S, flat)])


def screened(cell, P, v):
    """W~(R, i nu) on the kept entries from P(R, i nu) and v(q)."""
    n = len(cell.nu)
    Pq = to_dense(cell, "pb", n, P)
    eye = torch.eye(cell.NP, dtype=CD, device=DEV)
    for q in range(cell.nk):
        for i, j in _chunks(n, 4e7 / cell.NP ** 2):
            Pq[q, i:j] = torch.linalg.solve(eye - v[q] @ Pq[q, i:j], v[q].expand(j - i, -1, -1)) - v[q]
    return to_entries(cell, "pb", Pq)


def inverse_green(cell, H, Sx, S, mu, out=None):
    w = torch.from_numpy((2 * cell.om + 1) * np.pi / cell.beta).to(DEV)
    eye = torch.eye(cell.N, dtype=CD, device=DEV)
    return torch.linalg.inv((1j * w + mu)[None, :, None, None] * eye - (H + Sx)[:, None] - S)


def dyson_tau(cell, H, Sx, S, mu, rows=slice(None)):
    """G(k, tau) with the two leading tail terms carried exactly."""
    w = torch.from_numpy((2 * cell.om + 1) * np.pi / cell.beta).to(DEV)[None, :, None, None]
    T = torch.from_numpy(np.linalg.pinv(fourier(cell, "F"), rcond=1e-15)[rows]).to(DEV)
    t = torch.from_numpy(cell.tau[rows]).to(DEV)[None, :, None, None]
    eye = torch.eye(cell.N, dtype=CD, device=DEV)
    M1 = (H + Sx - mu * eye)[:, None]
    D = inverse_green(cell, H, Sx, S, mu) - eye / (1j * w) - M1 / (1j * w) ** 2
    G = torch.matmul(T[None], D.reshape(cell.nk, len(cell.om), -1)).view(cell.nk, -1, cell.N, cell.N)
    return G - 0.5 * eye + M1 * (2 * t - cell.beta) / 4


# ---- prepare, run, exact ------------------------------------------------------------------

def batch_cells(case, seed):
    out = []
    for i, text in enumerate(case["cells"].split(",")):
        c, mesh, cut = text.split("/")
        out.append(Cell(case, seed + i, text=c, mesh=mesh, cutoff=float(cut)))
    return out


def inputs(case, seed):
    """The cell and the seeded inputs of a case (nothing of the library is called)."""
    kind = case["kind"]
    if kind == "batch":
        cells = batch_cells(case, seed)
        return cells, dict(G_R=[to_entries(c, "orb", green(c, seed + i)) for i, c in enumerate(cells)],
                           W=[spread(c, "pb", _gen(seed, 20 + i), boson_tau(c)) for i, c in enumerate(cells)])
    cell = Cell(case, seed)
    g = _gen(seed)
    if kind == "sweep":
        return cell, dict(G_k=green(cell, seed), v_q=coulomb_q(cell, seed))
    if kind == "rows":
        return cell, dict(G_k=green(cell, seed), W_iw=spread(cell, "pb", g, boson_nu(cell)),
                          v_R=spread(cell, "pb", g, torch.ones(1, 1, dtype=CD, device=DEV)))
    if kind == "p":
        return cell, dict(G_R=to_entries(cell, "orb", green(cell, seed)))
    if kind == "sigma":
        return cell, dict(G_R=to_entries(cell, "orb", green(cell, seed)), W=spread(cell, "pb", g, boson_tau(cell)),
                          v_R=spread(cell, "pb", g, torch.ones(1, 1, dtype=CD, device=DEV)))
    if kind == "tau":
        return cell, dict(P=spread(cell, "pb", g, boson_tau(cell)), W_iw=spread(cell, "pb", g, boson_nu(cell)),
                          Sig=spread(cell, "orb", g, fermion_tau(cell)))
    if kind == "lattice":
        w = torch.from_numpy(1.0 / (1j * (2 * cell.om + 1) * np.pi / cell.beta - 0.3)).to(DEV)
        return cell, dict(G_k=green(cell, seed), v_q=coulomb_q(cell, seed).contiguous(),
                          Sig=spread(cell, "orb", g, w[None, :]))
    if kind == "w":
        P = polarizability(cell, to_entries(cell, "orb", green(cell, seed)))
        P = along(cell, "pb", fourier(cell, "B"), P)
        return cell, dict(P=torch.complex(P.real, torch.zeros_like(P.real)), v_q=coulomb_q(cell, seed).contiguous())
    H, e, _, mu = hamiltonian(cell, seed, 0.0)
    w = 1j * (2 * cell.om + 1) * np.pi / cell.beta
    S, Sx = self_energy_k(cell, seed, w)
    d = dict(H=H, Sx=Sx, S=S, mu=mu, lo=float(e.min()) - 1.0, hi=float(e.max()) + 1.0)
    if kind == "bands":
        d["w"] = np.linspace(-1.0, 1.0, case["n_real"])
        d["S_w"] = self_energy_k(cell, seed, d["w"] + 1j * case["delta"])[0]
    return cell, d


def prepare(case, seed):
    cell, s = inputs(case, seed)
    s["case"], s["cell"] = case, cell
    if case["kind"] == "batch":
        s["plans"] = [c.plan(defer_scratch=True) for c in cell]
        s["batch"] = gw.Batch(s["plans"])
    else:
        # only a program that solves for W holds that scratch
        s["plan"] = cell.plan(defer_scratch=case["kind"] not in ("sweep", "w", "p", "sigma") or case.get("precision") == "mixed",
                              **(dict(workspace_bytes=1 << 30) if case["kind"] in ("p", "sigma") else {}))
    if case["kind"] in ("rows", "tau"):
        # the frequencies nu < 0 of P are left as they are by the transform
        s["P_iw"] = torch.zeros(len(cell.nu) * cell.length("pb"), dtype=CD, device=DEV)
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "batch":
        return {"P": s["batch"].polarizability_tau(s["G_R"]), "Sigma": s["batch"].self_energy_tau(s["G_R"], s["W"])}
    p, cell = s["plan"], s["cell"]
    if kind == "sweep":
        G = p.green_k_to_R(s["G_k"].view(-1))
        P = p.polarizability_tau(G, precision=case["precision"])
        W = p.screened_W_iw(p.transform_tau_iw("B", "tau_to_iw", "pb", P), s["v_q"].view(-1))
        v_R = p.fourier_k_to_R("pb", 1, s["v_q"].view(-1))
        Wt = p.transform_tau_iw("B", "iw_to_tau", "pb", W)
        S, Sx = p.self_energy_tau(G, Wt, v_R=v_R, precision=case["precision"])
        return {"P": P, "W": W, "Sigma_k": p.fourier_R_to_k("orb", len(cell.om), p.transform_tau_iw("F", "tau_to_iw", "orb", S)),
                "Sigma_x": p.fourier_R_to_k("orb", 1, Sx)}
    if kind == "rows":
        G = p.green_k_to_R(s["G_k"].view(-1))
        P = p.polarizability_tau(G, precision=case["precision"])
        P_iw = p.transform_tau_iw("B", "tau_to_iw", "pb", P, out=s["P_iw"], structure="mirror_nonneg")
        del P
        W = p.transform_tau_iw("B", "iw_to_tau", "pb", s["W_iw"], structure="real")
        S, Sx = p.self_energy_tau(G, W, v_R=s["v_R"], precision=case["precision"])
        return {"P_iw": P_iw, "Sigma_k": p.fourier_R_to_k("orb", len(cell.om), p.transform_tau_iw("F", "tau_to_iw", "orb", S)),
                "Sigma_x": p.fourier_R_to_k("orb", 1, Sx)}
    if kind == "p":
        return p.polarizability_tau(s["G_R"], precision=case["precision"])
    if kind == "sigma":
        return list(p.self_energy_tau(s["G_R"], s["W"], v_R=s["v_R"], precision=case["precision"]))
    if kind == "tau":
        return {"P_iw": p.transform_tau_iw("B", "tau_to_iw", "pb", s["P"], out=s["P_iw"], structure="mirror_nonneg"),
                "W": p.transform_tau_iw("B", "iw_to_tau", "pb", s["W_iw"], structure="real"),
                "Sigma": p.transform_tau_iw("F", "tau_to_iw", "orb", s["Sig"])}
    if kind == "lattice":
        return {"G": p.green_k_to_R(s["G_k"].view(-1)), "v": p.fourier_k_to_R("pb", 1, s["v_q"].view(-1)),
                "Sigma_k": p.fourier_R_to_k("orb", len(cell.om), s["Sig"])}
    if kind == "w":
        return p.screened_W_iw(s["P"], s["v_q"].view(-1))
    H, Sx, S = s["H"].view(-1), s["Sx"].view(-1), s["S"].view(-1)
    if kind == "dyson":
        mu, n = p.chemical_potential(H, float(cell.N), s["lo"], s["hi"], Sigx_k=Sx, Sig_k_iw=S)
        return {"mu": mu, "n": n, "G": p.dyson_green_tau(H, mu, Sigx_k=Sx, Sig_k_iw=S)}
    return {"E": p.qp_energies(H, s["mu"], Sigx_k=Sx, Sig_k_iw=S),
            "Sigma_w": p.continue_sigma(S, s["w"], case["delta"]),
            "A": p.spectral_function(H, s["w"], case["delta"], s["mu"], Sigx_k=Sx, Sig_k_w=s["S_w"].view(-1))}


def _nonneg(cell, kind, P_iw):
    """The slices of nu >= 0, zeros elsewhere (the buffer that `run` hands over starts as zeros)."""
    keep = torch.from_numpy(cell.nu >= 0).to(DEV)[None, :, None, None]
    return join(cell, kind, len(cell.nu), [b * keep for b in split(cell, kind, len(cell.nu), P_iw)])


def exact(case, seed):
    kind = case["kind"]
    cell, s = inputs(case, seed)
    if kind == "batch":
        return {"P": [polarizability(c, G) for c, G in zip(cell, s["G_R"])],
                "Sigma": [sigma(c, G, W, c.nt) for c, G, W in zip(cell, s["G_R"], s["W"])]}
    n_om = len(cell.om)
    if kind == "p":
        return polarizability(cell, s["G_R"])
    if kind == "sigma":
        return [sigma(cell, s["G_R"], s["W"], cell.nt),
                sigma(cell, last_slice(cell, "orb", cell.nt, s["G_R"]), s["v_R"], 1, sign=1.0)]
    if kind == "lattice":
        return {"G": to_entries(cell, "orb", s["G_k"]), "v": to_entries(cell, "pb", s["v_q"][:, None]),
                "Sigma_k": to_dense(cell, "orb", n_om, s["Sig"]).reshape(-1)}
    if kind == "w":
        return screened(cell, s["P"], s["v_q"])
    if kind in ("tau", "rows", "sweep"):
        Tb, Tf = fourier(cell, "B"), fourier(cell, "F")
        Ti = np.linalg.pinv(Tb, rcond=1e-15)
    if kind == "tau":
        return {"P_iw": _nonneg(cell, "pb", along(cell, "pb", Tb, s["P"])), "W": along(cell, "pb", Ti, s["W_iw"]),
                "Sigma": along(cell, "orb", Tf, s["Sig"])}
    if kind in ("rows", "sweep"):
        G = to_entries(cell, "orb", s["G_k"])
        P = polarizability(cell, G)
        P_iw = along(cell, "pb", Tb, P)
        if kind == "rows":
            del P
            P_iw, v_R, W_iw = _nonneg(cell, "pb", P_iw), s["v_R"], s["W_iw"]
        else:
            v_R, W_iw = to_entries(cell, "pb", s["v_q"][:, None]), screened(cell, P_iw, s["v_q"])
        S = sigma(cell, G, along(cell, "pb", Ti, W_iw), cell.nt)
        Sx = sigma(cell, last_slice(cell, "orb", cell.nt, G), v_R, 1, sign=1.0)
        out = {"Sigma_k": to_dense(cell, "orb", n_om, along(cell, "orb", Tf, S)).reshape(-1),
               "Sigma_x": to_dense(cell, "orb", 1, Sx).reshape(-1)}
        return {**out, "P_iw": P_iw} if kind == "rows" else {**out, "P": P, "W": W_iw}
    if kind == "dyson":
        def count(mu):
            G = dyson_tau(cell, s["H"], s["Sx"], s["S"], mu, rows=slice(cell.nt - 1, cell.nt))
            return -2.0 * float(G.diagonal(dim1=-2, dim2=-1).sum().real) / cell.nk

        lo, hi = s["lo"], s["hi"]
        while hi - lo > 1e-12:
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if count(mid) < cell.N else (lo, mid)
        mu = 0.5 * (lo + hi)
        return {"mu": mu, "n": count(mu), "G": dyson_tau(cell, s["H"], s["Sx"], s["S"], mu).reshape(-1)}
    i0, i1 = int(np.nonzero(cell.om == 0)[0][0]), int(np.nonzero(cell.om == 1)[0][0])
    w0, w1 = np.pi / cell.beta, 3 * np.pi / cell.beta
    S1 = (s["S"][:, i1] - s["S"][:, i0]) / (1j * (w1 - w0))
    S0 = s["S"][:, i0] - 1j * w0 * S1
    herm = lambda x: 0.5 * (x + x.mH)  # noqa: E731
    eye = torch.eye(cell.N, dtype=CD, device=DEV)
    e, U = torch.linalg.eigh(eye - herm(S1))
    Ai = (U * e.rsqrt()[:, None, :]) @ U.mH
    E = torch.linalg.eigvalsh(herm(Ai @ (s["H"] + herm(s["Sx"]) + herm(S0) - s["mu"] * eye) @ Ai)) + s["mu"]
    z = torch.from_numpy(s["w"] + s["mu"] + 1j * case["delta"]).to(DEV)[None, :, None, None]
    G = torch.linalg.inv(z * eye - (s["H"] + s["Sx"])[:, None] - s["S_w"])
    A = -G.diagonal(dim1=-2, dim2=-1).sum(-1).imag / math.pi
    # the continued fraction has no value that 64 bits give to their own rounding
    return {"E": E.reshape(-1), "Sigma_w": None, "A": A.reshape(-1)}


def work(case):
    """Bytes: the inputs once and the outputs once; flops: the method's real operations."""
    kind = case["kind"]
    if kind == "batch":
        parts = [(c, Cell(case, 0, text=c.split("/")[0], mesh=c.split("/")[1], cutoff=float(c.split("/")[2])))
                 for c in case["cells"].split(",")]
        got = [_contraction(c, "p") for _, c in parts] + [_contraction(c, "sigma") for _, c in parts]
        return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}
    cell = Cell(case, 0)
    lo, lp = cell.length("orb"), cell.length("pb")
    n_om, n_nu, nt, half = len(cell.om), len(cell.nu), cell.nt, (cell.nt + 1) // 2
    pos = n_nu // 2 + 1
    nq = sum(1 if q == m else 0.5 for q, m in ((q, tuple((-x) % y for x, y in zip(q, cell.mesh))) for q in np.ndindex(*cell.mesh)))
    dense_o, dense_p = cell.nk * cell.N ** 2, cell.nk * cell.NP ** 2
    gather = (16 * (dense_o * nt + lo * nt), 2 * cell.nk * lo * nt)
    scatter = (16 * (dense_o * n_om + lo * n_om), 2 * cell.nk * lo * n_om)
    tau_p = (16 * lp * (half + pos), 4 * half * pos * lp)
    tau_w = (8 * lp * n_nu + 16 * lp * nt, 4 * n_nu * half * lp)
    tau_s = (16 * lo * (nt + n_om), 8 * nt * n_om * lo)
    solve = (8 * lp * pos + 16 * dense_p + 8 * lp * n_nu, 8.0 * cell.NP ** 3 * nq * pos)
    p, s = _contraction(cell, "p"), _contraction(cell, "sigma")
    inv = 8.0 * cell.N ** 3 * cell.nk
    parts = {"sweep": [gather, p, tau_p, solve, tau_w, s, tau_s, scatter], "rows": [gather, p, tau_p, tau_w, s, tau_s, scatter],
             "p": [p], "sigma": [s], "tau": [tau_p, tau_w, tau_s],
             "lattice": [gather, (16 * (dense_p + lp), 2 * cell.nk * lp), scatter], "w": [solve],
             "dyson": [(16 * dense_o * (n_om + nt + 2), inv * n_om + 8 * nt * n_om * dense_o)],
             "bands": [(16 * dense_o * 4, 3 * inv),
                       (16 * dense_o * (n_om // 2 + 2 * case.get("n_real", 0)), inv * case.get("n_real", 0))]}[kind]
    return {"bytes": float(sum(b for b, _ in parts)), "flops": float(sum(f for _, f in parts))}


def _contraction(cell, which):
    """(bytes, flops) of the P or Sigma contraction over the entries and nodes."""
    dims = cell.entries()[4]
    na, nb, Ka, Kb = (dims[k][i].astype(float) for k, i in (("orb", 0), ("orb", 1), ("pb", 0), ("pb", 1)))
    unit = 2 * (2 * Ka * na ** 2 * nb + 4 * Ka * na * nb ** 2 + 2 * Ka * Kb * nb ** 2)
    nodes = (cell.nt + 1) // 2 if which == "p" else cell.nt
    o, p = float((na * nb).sum()), float((Ka * Kb).sum())
    return (16 * cell.nt * (o + p), float(unit.sum()) * nodes) if which == "p" else (16 * cell.nt * (2 * o + p), float(unit.sum()) * nodes)
