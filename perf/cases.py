"""What the speed of this framework is measured on: one pass each of the calls its users make.

A case is a dict of plain values; ``prepare`` builds what a user's program holds before the call (basis,
Hamiltonian, vectors on the GPU), ``run`` is one call through the public entry points of
``paper_2505_02901_gb300.api`` and ``exact`` gives the same outputs from plain torch in 64 bits.

Kinds of calls
  apply     y = H x on a U(1) block, 1 to 8 right-hand sides: the step of every user-written iteration
  backward  y = H(J) x under autograd, then dL/dx and dL/dJ from a given dL/dy
  batch     one product on each of many small Hamiltonians, in one call
  evolve    exp(-iHt) psi (or exp(-tau H) psi), the whole call
  ftlm      finite-temperature Lanczos from several random starts, the whole call
  ground    ground energy and its gradient with respect to the couplings, the whole call
  sym       y = H x on a symmetry-adapted block
"""
import math

import numpy as np
import torch

from paper_2505_02901_gb300 import api, workloads as W

DEVICE = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # The smallest call: H x on the 16-site chain of a teaching or test script; one short launch, so latency.
        dict(name="apply_chain16_f64", kind="apply", lattice="chain", lx=16, ly=1, couplings="uniform", dn=0,
             dtype="f64", nvec=1),
        # A lattice of a size that people scan over parameters: odd numbers of rows, a cache-resident block.
        dict(name="apply_square4x5_f64", kind="apply", lattice="square", lx=4, ly=5, couplings="uniform", dn=0,
             dtype="f64", nvec=1),
        # The large product in full precision: the plain Lanczos iteration on the 4x8 J1-J2 lattice.
        dict(name="apply_square4x8_f64", kind="apply", lattice="square", lx=4, ly=8, couplings="uniform", dn=0,
             dtype="f64", nvec=1),
        # The same product with vectors stored in 32 bits, as long Lanczos runs on this lattice keep them.
        dict(name="apply_square4x8_f32", kind="apply", lattice="square", lx=4, ly=8, couplings="uniform", dn=0,
             dtype="f32", nvec=1),
        # Differentiation: forward and backward of the product on the 28-site ladder with its own coupling on
        # every bond (the training step of a fit of couplings).
        dict(name="backward_ladder28_f64", kind="backward", lattice="ladder", lx=14, ly=2, couplings="random",
             dtype="f64"),
        # Batching: 64 chains and ladders of uneven size, eight vectors each, in one call (disorder averages).
        dict(name="batch64x8_f32", kind="batch", count=64, nmin=18, nmax=28, dtype="f32", nvec=8),
        # Real-time evolution of an open ferromagnetic chain after a quench from a product state: complex vectors,
        # whole call.
        dict(name="evolve_chain24", kind="evolve", lattice="open", lx=24, ly=1, couplings="uniform", time=2.0,
             imaginary=False, start="product"),
        # Thermodynamics of the 4x6 J1-J2 lattice: eight random starts side by side, whole call.
        dict(name="ftlm_square4x6", kind="ftlm", lattice="square", lx=4, ly=6, couplings="uniform", starts=8,
             steps=30),
        # Ground energy of a small disordered ladder with dE/dJ: many short dependent steps, whole call.
        dict(name="ground_ladder16_f64", kind="ground", lattice="ladder", lx=8, ly=2, couplings="random",
             steps=120),
        # Symmetry-adapted blocks: the 36-site chain with translations and reflections (the dihedral group),
        dict(name="sym_chain36_dihedral", kind="sym", lattice="chain", lx=36, ly=1, group="dihedral", mx=0, my=0,
             dn=0),
        # the 6x6 J1-J2 lattice at momentum (pi/3, 0), whose vectors are complex,
        dict(name="sym_square6x6_k10", kind="sym", lattice="square", lx=6, ly=6, group="torus", mx=1, my=0, dn=0),
        # and the 6x6 triangular lattice with its whole space group (432 elements).
        dict(name="sym_triangular6x6_space", kind="sym", lattice="triangular", lx=6, ly=6, group="space", mx=0,
             my=0, dn=0),
    ]


def _lattice_upto(rng, nmin, nmax):
    """A lattice with nmin to nmax sites, its size spread evenly over the sites (the dimension's logarithm)."""
    n = rng.randint(nmin, nmax)
    kind = rng.choice(["chain", "ladder", "square", "triangular"])
    if kind == "square":
        fits = [(a, b) for a in (3, 4, 5) for b in range(3, 9) if nmin <= a * b <= nmax]
    elif kind == "triangular":
        fits = [(a, a) for a in (3, 4, 5) if nmin <= a * a <= nmax]
    elif kind == "ladder":
        fits = [(n // 2, 2)] if n // 2 >= 3 and 2 * (n // 2) >= nmin else []
    else:
        fits = []
    if not fits:
        return "chain", n, 1
    lx, ly = rng.choice(fits)
    return kind, lx, ly


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "backward", "batch", "evolve", "ftlm", "ground", "sym", "sym"])
    couplings = rng.choice(["uniform", "random"])
    if kind == "apply":
        nvec = rng.choice([1, 1, 1, 1, 2, 4, 8])
        lattice, lx, ly = _lattice_upto(rng, 10, 32 if nvec == 1 else 26)
        return dict(kind=kind, lattice=lattice, lx=lx, ly=ly, couplings=couplings, dn=rng.choice([0, 0, 1, 2, 3]),
                    dtype=rng.choice(["f64", "f32"]), nvec=nvec)
    if kind == "backward":
        lattice, lx, ly = _lattice_upto(rng, 10, 28)
        return dict(kind=kind, lattice=lattice, lx=lx, ly=ly, couplings=couplings, dtype=rng.choice(["f64", "f32"]))
    if kind == "batch":
        nvec = rng.choice([1, 2, 4, 8, 8])
        dtype = rng.choice(["f64", "f32"])
        nmax = rng.randint(12, 28 if (dtype, nvec) == ("f32", 8) else 22)
        return dict(kind=kind, count=round(4 * 16 ** rng.random()), nmin=rng.randint(8, nmax - 2), nmax=nmax,
                    dtype=dtype, nvec=nvec)
    if kind == "evolve":
        lattice, lx, ly = _lattice_upto(rng, 10, 24)
        if lattice == "chain" and rng.random() < 0.5:
            lattice = "open"
        return dict(kind=kind, lattice=lattice, lx=lx, ly=ly, couplings=couplings,
                    time=round(0.1 * 10 ** rng.random(), 3), imaginary=rng.random() < 0.25,
                    start=rng.choice(["product", "random"]))
    if kind == "ftlm":
        lattice, lx, ly = _lattice_upto(rng, 14, 24)
        return dict(kind=kind, lattice=lattice, lx=lx, ly=ly, couplings=couplings, starts=rng.randint(1, 16),
                    steps=rng.randint(8, 24))
    if kind == "ground":
        n = rng.randint(10, 22)  # even rings: a unique ground state
        lattice, lx, ly = ("ladder", 2 * (n // 4), 2) if n >= 12 and rng.random() < 0.5 else ("chain", n - n % 2, 1)
        return dict(kind=kind, lattice=lattice, lx=lx, ly=ly, couplings=couplings, steps=120)
    group = rng.choice(["translations", "dihedral", "torus", "torus", "space"])
    dn = rng.choice([0, 0, 1, 2])
    if group in ("translations", "dihedral"):
        n = rng.randint(12, 34)
        return dict(kind=kind, lattice="chain", lx=n, ly=1, group=group, dn=dn, my=0,
                    mx=0 if group == "dihedral" else rng.choice([0, 1, n // 2]))
    if group == "torus":
        lx, ly = rng.choice([(4, 4), (3, 6), (4, 5), (3, 7), (4, 6), (5, 5), (5, 6), (4, 7), (6, 6)])
        return dict(kind=kind, lattice="square", lx=lx, ly=ly, group=group, mx=rng.choice([0, 0, 1]),
                    my=rng.choice([0, 1]), dn=dn if lx * ly < 36 else dn + 3)
    lattice, lx = rng.choice([("square", 4), ("square", 5), ("square", 6), ("triangular", 4), ("triangular", 5),
                              ("triangular", 6)])
    return dict(kind=kind, lattice=lattice, lx=lx, ly=lx, group=group, mx=0, my=0, dn=dn)


# ----------------------------------------------------------------- inputs
def _sites(case):
    return case["lx"] * case["ly"]


def _graph(case, seed):
    """(bonds, J) of the case's lattice; random couplings are uniform in [0.5, 1.5)."""
    lattice, lx, ly = case["lattice"], case["lx"], case["ly"]
    if lattice == "chain":
        bonds = W.chain(lx)
        J = np.ones(len(bonds))
    elif lattice == "open":
        bonds = np.array([(i, i + 1) for i in range(lx - 1)], dtype=np.int32)
        J = -np.ones(len(bonds))
    elif lattice == "ladder":
        bonds = W.ladder(lx, 2)
        J = np.ones(len(bonds))
    elif lattice == "square":
        bonds, J = W.square_j1j2(lx, ly, 1.0, 0.5)
    else:
        bonds, J = W.triangular(lx)
    if case.get("couplings") == "random":
        J = W.uniform_couplings(len(bonds), seed)
    return bonds, np.asarray(J, dtype=np.float64)


def _symmetry(case):
    group, lx, ly, mx, my = case["group"], case["lx"], case["ly"], case["mx"], case["my"]
    if group == "translations":
        return W.chain_translations(lx), W.chain_characters(lx, mx)
    if group == "dihedral":
        return W.chain_dihedral(lx), W.chain_dihedral_characters(lx, mx, 1)
    if group == "torus":
        return W.torus_translations(lx, ly), W.torus_characters(lx, ly, mx, my)
    return W.space_group(lx, ly, case["lattice"]), W.space_group_characters(lx, ly, case["lattice"])


def _nup(case):
    n = _sites(case)
    return n // 2 - min(case.get("dn", 0), n // 2 - 1)


def _dtype(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.float64


def _normal(shape, dtype, seed, stream):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(1000 * seed + stream)
    return torch.randn(shape, dtype=dtype, device=DEVICE, generator=g)


def _vector(case, dim, seed, stream):
    nvec = case.get("nvec", 1)
    return _normal((dim,) if nvec == 1 else (dim, nvec), _dtype(case), seed, stream)


def _instances(case, seed):
    """The chains and ladders of a batch: even sizes from nmin to nmax, each with its own couplings.

    The sizes and kinds belong to the case, the couplings to the seed."""
    shape = np.random.default_rng(1000 * case["count"] + 10 * case["nmin"] + case["nmax"])
    sizes = [n for n in range(case["nmin"], case["nmax"] + 1) if n % 2 == 0]
    out = []
    for k in range(case["count"]):
        n = int(shape.choice(sizes))
        ladder = bool(shape.integers(0, 2)) and n >= 6
        bonds = W.ladder(n // 2, 2) if ladder else W.chain(n)
        out.append((n, bonds, W.uniform_couplings(len(bonds), 100 * seed + k)))
    return out


def _start(case, seed):
    """Unit start vector of an evolution: a product state of half the spins up (one basis word) or a random state."""
    n = _sites(case)
    dim = math.comb(n, n // 2)
    psi = torch.zeros(dim, dtype=torch.complex128, device=DEVICE)
    if case["start"] == "product":
        psi[np.random.default_rng(seed).integers(dim)] = 1.0
    else:
        z = _normal((dim, 2), torch.float64, seed, 1)
        psi = torch.view_as_complex(z / z.norm())
    return psi


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case)
    if kind == "batch":
        hams, xs = [], []
        for k, (n, bonds, J) in enumerate(_instances(case, seed)):
            hams.append(api.Hamiltonian(api.Basis(n, n // 2, bonds), J))
            xs.append(_vector(case, hams[-1].dim, seed, 10 + k))
        return dict(state, hams=hams, xs=xs, ys=[torch.empty_like(x) for x in xs])
    bonds, J = _graph(case, seed)
    basis = api.Basis(_sites(case), _nup(case), bonds, _symmetry(case) if kind == "sym" else None)
    state["ham"] = ham = api.Hamiltonian(basis, J)
    if kind == "apply":
        state["x"] = _vector(case, ham.dim, seed, 1)
        state["y"] = torch.empty_like(state["x"])
    elif kind == "sym":
        x = _normal((ham.dim, 2) if basis.is_complex else (ham.dim,), torch.float64, seed, 1)
        state["x"] = torch.view_as_complex(x) if basis.is_complex else x
        state["y"] = torch.empty_like(state["x"])
    elif kind == "backward":
        state["J"] = torch.tensor(J, requires_grad=True)
        state["x"] = _vector(case, ham.dim, seed, 1).requires_grad_()
        state["g"] = _vector(case, ham.dim, seed, 2)
    elif kind == "evolve":
        state["psi"] = _start(case, seed)
    elif kind == "ftlm":
        state["seed"] = seed + 1
    elif kind == "ground":
        state["J"] = torch.tensor(J, requires_grad=True)
        state["seed"] = seed + 1
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("apply", "sym"):
        return state["ham"].apply(state["x"], out=state["y"])
    if kind == "backward":
        J, x = state["J"], state["x"]
        y = api.heisenberg_apply(state["ham"], J, x)
        gJ, gx = torch.autograd.grad(y, (J, x), state["g"])
        return y.detach(), gx, gJ
    if kind == "batch":
        api.batch_apply(state["hams"], state["xs"], state["ys"])
        return state["ys"]
    if kind == "evolve":
        t = case["time"]
        psi, _ = state["ham"].evolve(state["psi"], t=0.0 if case["imaginary"] else t,
                                     tau=t if case["imaginary"] else 0.0, max_iter=300, tol=1e-12)
        return psi
    if kind == "ftlm":
        alpha, beta, _ = state["ham"].ftlm(case["starts"], case["steps"], state["seed"])
        return alpha, beta
    e0 = api.ground_energy(state["ham"], state["J"], max_iter=case["steps"], seed=state["seed"])
    (gJ,) = torch.autograd.grad(e0, state["J"])
    return e0.detach(), gJ


# ------------------------------------------------------------------- work
def _flips(n, nup, nb):
    """Mean number of antiparallel bonds of a state: the off-diagonal elements of a row."""
    return nb * 2.0 * nup * (n - nup) / (n * (n - 1))


def work(case):
    """Compulsory bytes (inputs read once, outputs written once) and multiply-adds of a pass."""
    kind = case["kind"]
    esize = 4 if case.get("dtype") == "f32" else 8
    if kind == "batch":
        nbytes = flops = 0
        for n, bonds, _ in _instances(case, 0):
            cells = math.comb(n, n // 2) * case["nvec"]
            nbytes += 2 * esize * cells
            flops += 2 * cells * (1 + _flips(n, n // 2, len(bonds)))
        return dict(bytes=nbytes, flops=flops)
    bonds, J = _graph(case, 0)
    n, nup, nb = _sites(case), _nup(case), len(bonds)
    dim, per_row = math.comb(n, nup), 1 + _flips(n, nup, nb)
    if kind == "apply":
        cells = dim * case["nvec"]
        return dict(bytes=2 * esize * cells, flops=2 * cells * per_row)
    if kind == "sym":
        perms, chi = _symmetry(case)
        parts = 2 if np.abs(np.asarray(chi).imag).max() > 1e-12 else 1
        rows = dim // len(perms)
        return dict(bytes=2 * 8 * parts * rows, flops=2 * parts * rows * per_row)
    if kind == "backward":  # y = H x; gx = H g; one sum per bond
        return dict(bytes=5 * esize * dim, flops=2 * dim * (2 * per_row + per_row + nb))
    if kind == "ftlm":  # a step reads two vectors and writes one
        steps = 8 * ((case["starts"] + 7) // 8) * case["steps"]
        return dict(bytes=3 * 8 * dim * steps, flops=2 * dim * steps * (per_row + 4))
    if kind == "ground":  # two passes of the recurrence, then one sum per bond
        return dict(bytes=2 * 3 * 8 * dim * case["steps"], flops=2 * dim * (2 * case["steps"] * (per_row + 4) + nb))
    # evolution: two passes of as many steps as the spectral width times the time needs, on complex vectors
    steps = int(10 + 0.5 * case["time"] * float(np.abs(J).sum()))
    return dict(bytes=2 * 3 * 16 * dim * steps, flops=2 * 2 * dim * 2 * steps * (per_row + 4))


# ------------------------------------------------ the same in plain 64 bits
class _Block:
    """Words of n bits with nup ones in ascending order, on the GPU, and their ranks by two tables."""

    def __init__(self, n, nup):
        self.n, self.nup, self.L = n, nup, min(n // 2, 14)
        lo = np.arange(1 << self.L)
        lo_pop = np.array([int(v).bit_count() for v in lo])
        order = np.lexsort((lo, lo_pop))
        first = np.searchsorted(lo_pop[order], np.arange(self.L + 2))
        rank = np.empty(len(lo), dtype=np.int64)
        rank[order] = np.arange(len(lo)) - first[lo_pop[order]]
        hi = torch.arange(1 << (n - self.L), device=DEVICE)
        need = nup - sum((hi >> b) & 1 for b in range(n - self.L))
        size = torch.tensor([math.comb(self.L, m) for m in range(self.L + 1)], device=DEVICE)
        ok = (need >= 0) & (need <= self.L)
        count = torch.where(ok, size[need.clamp(0, self.L)], torch.zeros_like(need))
        self.hi_off = torch.cumsum(count, 0) - count
        self.dim = int(count.sum())
        self.rank = torch.from_numpy(rank).to(DEVICE)
        self.order = torch.from_numpy(order.astype(np.int64)).to(DEVICE)
        self.first = torch.from_numpy(first.astype(np.int64)).to(DEVICE)[need.clamp(0, self.L)]

    def words(self, r0, r1):
        r = torch.arange(r0, r1, device=DEVICE)
        h = torch.searchsorted(self.hi_off, r, right=True) - 1
        return (h << self.L) | self.order[self.first[h] + r - self.hi_off[h]]

    def index(self, s):
        return self.hi_off[s >> self.L] + self.rank[s & ((1 << self.L) - 1)]


_CHUNK = 1 << 24


def _flipped(s, i, j):
    """The word with the spins of sites i and j exchanged."""
    t = ((s >> i) ^ (s >> j)) & 1
    return s ^ (t * ((1 << i) | (1 << j)))


def _apply64(block, bonds, J, x, g=None):
    """H x, and with g also g . (S_i S_j x) for every bond: S_i S_j = P_ij / 2 - 1 / 4."""
    y = torch.empty_like(x)
    dots = torch.zeros(len(bonds), dtype=torch.float64, device=DEVICE)
    for r0 in range(0, block.dim, _CHUNK):
        r1 = min(block.dim, r0 + _CHUNK)
        s, xc = block.words(r0, r1), x[r0:r1]
        acc = -0.25 * float(np.sum(J)) * xc
        for b, (i, j) in enumerate(bonds.tolist()):
            px = x[block.index(_flipped(s, i, j))]
            acc += 0.5 * float(J[b]) * px
            if g is not None:
                dots[b] += (g[r0:r1] * (0.5 * px - 0.25 * xc)).sum()
        y[r0:r1] = acc
    return y if g is None else (y, dots)


class _Fast:
    """The product as stored gathers, for calls that need many of them."""

    def __init__(self, block, bonds, J):
        s = block.words(0, block.dim)
        self.J, self.to = J, [block.index(_flipped(s, i, j)).to(torch.int32) for i, j in bonds.tolist()]

    def __call__(self, x):
        y = -0.25 * float(np.sum(self.J)) * x
        for c, to in zip(self.J, self.to):
            y += 0.5 * float(c) * x[to]
        return y

    def dots(self, x):
        return torch.stack([(x * (0.5 * x[to] - 0.25 * x)).sum() for to in self.to])


def _exact_sym(case, seed):
    """B^H H B x: x lifted to the U(1) block, the U(1) product, the rows of the representatives."""
    perms, chi = _symmetry(case)
    chi = np.asarray(chi, dtype=np.complex128)
    n, block = _sites(case), _Block(_sites(case), _nup(case))
    if block.dim * len(perms) * n > 5e10:
        return None
    bonds, J = _graph(case, seed)
    s = block.words(0, block.dim)
    rep, which = s.clone(), torch.zeros_like(s)
    stab = torch.zeros_like(s)
    overlap = torch.zeros(block.dim, dtype=torch.complex128, device=DEVICE)
    for g, p in enumerate(np.asarray(perms).tolist()):
        image = torch.zeros_like(s)
        for i, pi in enumerate(p):
            image |= ((s >> pi) & 1) << i
        same, less = image == s, image < rep
        stab += same
        overlap += same * complex(chi[g])
        which = torch.where(less, torch.full_like(which, g), which)
        rep = torch.minimum(rep, image)
    identity = [g for g, p in enumerate(np.asarray(perms).tolist()) if p == sorted(p)][0]
    which = torch.where(rep == s, torch.full_like(which, identity), which)
    member = overlap.abs() > 1e-9 * stab
    rows = torch.nonzero((rep == s) & member)[:, 0]
    place = torch.cumsum((rep == s) & member, 0) - 1
    cplx = bool(np.abs(chi.imag).max() > 1e-12)
    x = _normal((len(rows), 2) if cplx else (len(rows),), torch.float64, seed, 1)
    x = torch.view_as_complex(x) if cplx else x.to(torch.complex128)
    norm = (stab.to(torch.float64) / len(perms)).sqrt()
    at = block.index(rep)
    weight = torch.from_numpy(chi).to(DEVICE)[which] * norm * member[at]
    v = x[place[at].clamp(min=0)] * weight
    y = _apply64(block, bonds, J, v)[rows] / norm[rows]
    return y if cplx else y.real.contiguous()


def _exact_evolve(case, seed):
    """Taylor series of the exponential in steps of norm below one."""
    bonds, J = _graph(case, seed)
    n = _sites(case)
    H = _Fast(_Block(n, n // 2), bonds, J)
    psi = _start(case, seed)
    steps = max(1, math.ceil(case["time"] * 0.75 * float(np.abs(J).sum())))
    z = case["time"] / steps * (1.0 if case["imaginary"] else 1j)
    for _ in range(steps):
        term = psi
        for k in range(1, 19):
            term = H(term) * (-z / k)
            psi = psi + term
    return psi


def _splitmix(z):
    def srl(v, s):
        return (v >> s) & ((1 << (64 - s)) - 1)

    def wrap(c):
        return c - (1 << 64) if c >= 1 << 63 else c
    z = z + wrap(0x9E3779B97F4A7C15)
    z = (z ^ srl(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ srl(z, 27)) * wrap(0x94D049BB133111EB)
    return z ^ srl(z, 31)


def _seeded_normal(dim, seed):
    """The seeded start vector of the Lanczos calls, by its published definition (SplitMix64, Box-Muller)."""
    gamma = 0x9E3779B97F4A7C15 - (1 << 64)
    c = _splitmix(torch.tensor([seed], device=DEVICE)) + 2 * torch.arange(dim, device=DEVICE) * gamma

    def uniform(z):
        return (((_splitmix(z) >> 11) & ((1 << 53) - 1)).to(torch.float64) + 1.0) * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(uniform(c))) * torch.cos(2.0 * math.pi * uniform(c + gamma))


def _exact_ftlm(case, seed):
    bonds, J = _graph(case, seed)
    n = _sites(case)
    block = _Block(n, n // 2)
    H = _Fast(block, bonds, J)
    alpha, beta = np.zeros((2, case["starts"], case["steps"]))
    for r in range(case["starts"]):
        u = _seeded_normal(block.dim, seed + 1 + r)
        u = u / u.norm()
        before, b = torch.zeros_like(u), 0.0
        for k in range(case["steps"]):
            w = H(u) - b * before
            a = float(torch.dot(w, u))
            w = w - a * u
            b = float(w.norm())
            alpha[r, k], beta[r, k] = a, b
            before, u = u, w / b
    return alpha, beta


def _exact_ground(case, seed):
    """Lanczos with full reorthogonalisation, restarted from its own Ritz vector."""
    bonds, J = _graph(case, seed)
    n = _sites(case)
    block = _Block(n, n // 2)
    if block.dim > 200000:
        return None
    H = _Fast(block, bonds, J)
    v = _normal((block.dim,), torch.float64, seed, 3)
    for _ in range(3):
        V = torch.zeros((min(120, block.dim), block.dim), dtype=torch.float64, device=DEVICE)
        V[0] = v / v.norm()
        m = V.shape[0]
        for k in range(m - 1):
            w = H(V[k])
            for _twice in range(2):
                w = w - V[: k + 1].T @ (V[: k + 1] @ w)
            if float(w.norm()) < 1e-10:
                m = k + 1
                break
            V[k + 1] = w / w.norm()
        T = torch.stack([V[:m] @ H(V[k]) for k in range(m)])
        _, q = torch.linalg.eigh(0.5 * (T + T.T))
        v = q[:, 0] @ V[:m]
    v = v / v.norm()
    return torch.dot(v, H(v)).cpu(), H.dots(v).cpu()


def exact(case, seed):
    kind = case["kind"]
    if kind == "sym":
        return _exact_sym(case, seed)
    if kind == "evolve":
        return _exact_evolve(case, seed)
    if kind == "ftlm":
        return _exact_ftlm(case, seed)
    if kind == "ground":
        return _exact_ground(case, seed)
    if kind == "batch":
        return [_apply64(_Block(n, n // 2), bonds, J, _vector(case, math.comb(n, n // 2), seed, 10 + k).double())
                for k, (n, bonds, J) in enumerate(_instances(case, seed))]
    bonds, J = _graph(case, seed)
    block = _Block(_sites(case), _nup(case))
    x = _vector(case, block.dim, seed, 1).double()
    if kind == "apply":
        return _apply64(block, bonds, J, x)
    g = _vector(case, block.dim, seed, 2).double()
    y, dots = _apply64(block, bonds, J, x, g)
    return y, _apply64(block, bonds, J, g), dots.cpu()
