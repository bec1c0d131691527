"""Measured cases: what a user of this library has it do, from one product on a few thousand
rows to fused solver steps on billions of them.

A case is one call of the Python binding (apply_H, lanczos, lanczos_sectors, tpq,
inverse_iteration) on a lattice model.  `prepare` builds the model and the vectors a program
holds before the call, `run` is the call, `exact` restates it in 64-bit torch arithmetic.

Results that the library computes from single-precision vectors (the records of an fp32 run)
are returned as single-precision numbers, which is what such a run claims; the fp64
Rayleigh quotient of a refined run stays fp64.
"""
import math

import numpy as np
import torch

import paper_1703_03637_gb300 as hp

PRECS = {"fp64": hp.FP64, "fp32": hp.FP32}


# ------------------------------------------------------------------------------- lattices
def _ring(n, dist=1):
    return sorted({(min(i, (i + dist) % n), max(i, (i + dist) % n)) for i in range(n) if (i + dist) % n != i})


def _square(lx, ly):
    seen = []
    for y in range(ly):
        for x in range(lx):
            for dx, dy in ((1, 0), (0, 1)):
                a, b = x + lx * y, (x + dx) % lx + lx * ((y + dy) % ly)
                if a != b and (min(a, b), max(a, b)) not in seen:
                    seen.append((min(a, b), max(a, b)))
    return seen


def _honeycomb(cx, cy):
    seen = []
    for y in range(cy):
        for x in range(cx):
            a = 2 * (x + cx * y)
            for axis, (bx, by) in ((2, (x, y)), (0, (x - 1, y)), (1, (x, y - 1))):
                b = 2 * (bx % cx + cx * (by % cy)) + 1
                if (min(a, b), max(a, b), axis) not in seen:
                    seen.append((min(a, b), max(a, b), axis))
    return seen


def _tilted(w):
    """The periodic square cluster of 2 w^2 sites spanned by (w, w) and (-w, w)."""
    n, site = 2 * w * w, {}

    def key(x, y):
        return ((x * w + y * w) % n, (y * w - x * w) % n)

    cells = [(x, y) for y in range(-2 * w, 2 * w + 1) for x in range(-2 * w, 2 * w + 1)]
    at = [c for c in cells if key(*c) not in site and site.setdefault(key(*c), len(site)) is not None]
    bonds = []
    for i, (x, y) in enumerate(at):
        for dx, dy in ((1, 0), (0, 1)):
            j = site[key(x + dx, y + dy)]
            if i != j and (min(i, j), max(i, j)) not in bonds:
                bonds.append((min(i, j), max(i, j)))
    return n, bonds


def _terms(c):
    """Sites, couplings (i, j, 3x3 J), fields (hx, hy, hz) on every site, hopping bonds, t, U."""
    m = c["model"]
    none = (0.0, 0.0, 0.0)
    if m == "heisenberg_ring":
        return c["n"], [(i, j, np.eye(3)) for i, j in _ring(c["n"])], none, [], 0.0, 0.0
    if m == "heisenberg_square":
        return c["lx"] * c["ly"], [(i, j, np.eye(3)) for i, j in _square(c["lx"], c["ly"])], none, [], 0.0, 0.0
    if m == "j1j2_ring":
        cp = [(i, j, np.eye(3)) for i, j in _ring(c["n"])] + [(i, j, 0.5 * np.eye(3)) for i, j in _ring(c["n"], 2)]
        return c["n"], cp, none, [], 0.0, 0.0
    if m == "xxz_dm_ring":  # S^z-conserving with complex exchange: J^xy = -J^yx
        J = np.array([[1.0, 0.3, 0.0], [-0.3, 1.0, 0.0], [0.0, 0.0, 0.7]])
        return c["n"], [(i, j, J) for i, j in _ring(c["n"])], none, [], 0.0, 0.0
    if m == "kitaev_honeycomb":
        cp = []
        for i, j, a in _honeycomb(c["cx"], c["cy"]):
            J = np.zeros((3, 3))
            J[a, a] = -1.0
            cp.append((i, j, J))
        return 2 * c["cx"] * c["cy"], cp, (0.05, 0.05, 0.05), [], 0.0, 0.0
    if m == "hubbard_tilted":
        n, bonds = _tilted(c["w"])
        return n, [], none, bonds, 1.0, 8.0
    if m == "hubbard_square":
        return c["lx"] * c["ly"], [], none, _square(c["lx"], c["ly"]), 1.0, 8.0
    if m == "hubbard_ring":
        return c["n"], [], none, _ring(c["n"]), 1.0, 8.0
    raise KeyError(m)


def _model(c):
    n, couplings, h, bonds, t, U = _terms(c)
    m = hp.Model(hp.HUBBARD if bonds else hp.SPIN_HALF, n)
    for i, j, J in couplings:
        m.add_spin_coupling(i, j, J)
    if any(h):
        for i in range(n):
            m.add_spin_field(i, h)
    for i, j in bonds:
        for s in (0, 1):
            m.add_hopping(i, j, s, t)
    if U:
        for i in range(n):
            m.add_onsite_U(i, U)
    if bonds:
        m.set_basis(hp.BASIS_NUMBER, c["n_up"], c["n_dn"])
    elif "n_up" in c:
        m.set_basis(hp.BASIS_SZ, c["n_up"])
    else:
        m.set_basis(hp.BASIS_FULL)
    m.build()
    return m


def _rows(c):
    n, _, _, bonds, _, _ = _terms(c)
    if bonds:
        return math.comb(n, c["n_up"]) * math.comb(n, c["n_dn"])
    return math.comb(n, c["n_up"]) if "n_up" in c else 1 << n


def _complex(c):
    return c["model"] in ("kitaev_honeycomb", "xxz_dm_ring")


def _gauss(c, seed, rows, nvec):
    """A program's own normal vector, fp64, in shape [rows, nvec]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn((rows, nvec * (2 if _complex(c) else 1)), generator=g, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(v.view(rows, nvec, 2)) if _complex(c) else v


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # One product on the smallest cluster the paper checks itself with (8 sites, half
        # filling): an outside eigensolver or a time evolution calls this in a loop, so its
        # launches and its host path are what it waits for.
        dict(name="hubbard8_apply", call="apply", model="hubbard_tilted", w=2, n_up=4, n_dn=4, nvec=1, prec="fp64"),
        # A whole ground-state search on the 12-site ring, the first thing a new user runs.
        dict(name="ring12_lanczos", call="lanczos", model="heisenberg_ring", n=12, steps=24, prec="fp64"),
        # Inverse iteration on a mid-size cluster (2.7 million rows): products and streaming
        # vector kernels of a few microseconds each, hundreds of launches.
        dict(name="square24_cg", call="invit", model="heisenberg_square", lx=6, ly=4, n_up=12, steps=32),
        # Complex exchange in an S^z sector (Dzyaloshinskii-Moriya rings): the generic kernels.
        dict(name="xxz_dm22_lanczos", call="lanczos", model="xxz_dm_ring", n=22, n_up=11, steps=10, prec="fp64"),
        # mTPQ with 64 complex fp64 starts and observables on 18 sites, the accurate form of
        # the finite-temperature run.
        dict(name="kitaev18_tpq64", call="tpq", model="kitaev_honeycomb", cx=3, cy=3, starts=64, steps=4, obs=2,
             l=1.0, prec="fp64"),
        # Every S^z sector of the 28-site J1-J2 ring in one call: tiny and large sectors together.
        dict(name="j1j2_28_sectors", call="sectors", model="j1j2_ring", n=28, steps=10, prec="fp64"),
        # The main path, ground state of a square-lattice antiferromagnet in fp64 (6x5 torus,
        # S^z = 0, 155 million rows), a short stretch of its Lanczos steps.
        dict(name="square30_lanczos", call="lanczos", model="heisenberg_square", lx=6, ly=5, n_up=15, steps=8,
             prec="fp64"),
        # The same in fp32 with the fp64 refinement of energy and residual.
        dict(name="square30_refined", call="refined", model="heisenberg_square", lx=6, ly=5, n_up=15, steps=8,
             prec="fp32"),
        # Half-filled 4x4 Hubbard model, 166 million rows, fp64 Lanczos steps.
        dict(name="hubbard16_lanczos", call="lanczos", model="hubbard_square", lx=4, ly=4, n_up=8, n_dn=8, steps=8,
             prec="fp64"),
        # One fp32 product away from half filling, up and down rows of different, odd lengths.
        dict(name="hubbard16_apply32", call="apply", model="hubbard_square", lx=4, ly=4, n_up=7, n_dn=6, nvec=1,
             prec="fp32"),
        # 64 fp32 starts on the 24-site Kitaev cluster: the widest blocks (2^24 rows x 64).
        dict(name="kitaev24_tpq64", call="tpq", model="kitaev_honeycomb", cx=4, cy=3, starts=64, steps=2, obs=0,
             l=1.0, prec="fp32"),
        # The paper's 18-site Hubbard mTPQ, S^z = 0: 2.4 billion rows in fp32.
        dict(name="hubbard18_tpq", call="tpq", model="hubbard_tilted", w=3, n_up=9, n_dn=9, starts=1, steps=2, obs=0,
             l=8.0, prec="fp32"),
    ]


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["spin_sector", "spin_sector", "hubbard", "hubbard", "kitaev", "sectors", "complex"])
    prec = rng.choice(["fp64", "fp32"])
    if kind == "spin_sector":
        lat = rng.choice(["heisenberg_ring", "j1j2_ring", "heisenberg_square"])
        if lat == "heisenberg_square":
            lx, ly = rng.choice([(4, 3), (4, 4), (5, 4), (6, 4), (5, 5), (7, 4), (6, 5), (10, 3)])
            n, c = lx * ly, dict(model=lat, lx=lx, ly=ly)
        else:
            n = rng.randint(12, 30)
            c = dict(model=lat, n=n)
        c["n_up"] = max(3, min(n // 2, n // 2 - int(rng.expovariate(0.6))))
        call = rng.choice(["apply", "lanczos", "lanczos", "refined", "invit"])
        if call == "apply":
            return dict(call=call, **c, nvec=rng.choice([1, 1, 1, 2, 3, 5]) if math.comb(n, c["n_up"]) < 2e7 else 1,
                        prec=prec)
        if call == "invit":
            return dict(call=call, **c, steps=rng.randint(4, 24))
        return dict(call=call, **c, steps=rng.randint(4, 10), prec="fp32" if call == "refined" else prec)
    if kind == "hubbard":
        if rng.random() < 0.5:
            c = dict(model="hubbard_square", lx=4, ly=rng.choice([3, 4]))
            n = 4 * c["ly"]
        else:
            n = rng.randint(6, 14)
            c = dict(model="hubbard_ring", n=n)
        c.update(n_up=rng.randint(2, n // 2), n_dn=rng.randint(2, n // 2))
        call = rng.choice(["apply", "lanczos", "tpq", "refined"])
        if call == "apply":
            return dict(call=call, **c, nvec=1, prec=prec)
        if call == "tpq":
            return dict(call=call, **c, starts=1, steps=rng.randint(2, 8), obs=rng.choice([0, 2]), l=8.0, prec=prec)
        return dict(call=call, **c, steps=rng.randint(4, 8), prec="fp32" if call == "refined" else prec)
    if kind == "kitaev":
        cx, cy = rng.choice([(3, 2), (4, 2), (3, 3), (5, 2), (6, 2), (4, 3)])
        most = {6: 256, 8: 256, 9: 128, 10: 128, 12: 32}[cx * cy]
        starts = 1 << rng.randint(0, int(math.log2(most)))
        c = dict(model="kitaev_honeycomb", cx=cx, cy=cy)
        if rng.random() < 0.4:
            return dict(call="apply", **c, nvec=starts, prec=prec)
        return dict(call="tpq", **c, starts=starts, steps=rng.randint(2, 4), obs=rng.choice([0, 2]), l=1.0, prec=prec)
    if kind == "sectors":
        return dict(call="sectors", model="j1j2_ring", n=rng.randint(16, 26), steps=rng.randint(4, 8), prec=prec)
    n = rng.randint(12, 24)
    return dict(call=rng.choice(["apply", "lanczos"]), model="xxz_dm_ring", n=n, n_up=n // 2 - rng.randint(0, 2), nvec=1,
                steps=rng.randint(4, 8), prec=prec)


def _cg_energy(c):
    """A few couplings below the antiferromagnet's ground state, as a converged energy less its error is."""
    n, couplings, _, _, _, _ = _terms(c)
    return -0.36 * sum(J[2, 2] for _, _, J in couplings) - 0.1 * n


def prepare(case, seed):
    c = dict(case)
    m = _model(c)
    s = dict(c=c, m=m, seed=seed)
    if c["call"] == "apply":
        s["v"] = _gauss(c, seed, m.dim, c["nvec"]).to(m.dtype(PRECS[c["prec"]]))
        s["w"] = torch.empty_like(s["v"])
    elif c["call"] == "invit":
        s["x"] = _gauss(c, seed, m.dim, 1)[:, 0].contiguous()
        s["y"] = torch.empty_like(s["x"])
    return s


def _record(x, prec):
    return np.asarray(x, dtype=np.float32 if prec == "fp32" else np.float64)


def run(s):
    c, m = s["c"], s["m"]
    call = c["call"]
    if call == "apply":
        return m.apply_H(s["v"], s["w"])
    if call == "invit":
        s["y"].copy_(s["x"])  # the solve works in place; the program keeps its vector
        r = m.inverse_iteration(s["y"], _cg_energy(c), shift=0.1, outer=1, max_cg=c["steps"])
        return dict(x=s["y"], e=np.float64(r["e"]))
    prec = PRECS[c["prec"]]
    if call == "sectors":
        r = m.lanczos_sectors(list(range(c["n"] + 1)), c["steps"], prec=prec, seed=s["seed"])
        return {k: _record(np.concatenate([x[k] for x in r]), c["prec"]) for k in ("alpha", "beta", "eig")}
    if call in ("lanczos", "refined"):
        r = m.lanczos(c["steps"], prec=prec, seed=s["seed"], refine=call == "refined")
        out = {k: _record(r[k], c["prec"]) for k in ("alpha", "beta", "eig")}
        if call == "refined":
            out.update(e=np.float64(r["e_refined"]), residual=_record(r["residual"], c["prec"]),
                       variance=_record(r["variance"], c["prec"]))
        return out
    r = m.tpq(c["starts"], c["steps"], l=c["l"], prec=prec, seed=s["seed"], obs_every=c["obs"])
    return {k: _record(r[k], c["prec"]) for k in ("u", "h2", "norm", "doublon", "sz", "sz2")[:6 if c["obs"] else 3]}


# ------------------------------------------------------------------------------- work
def work(case):
    """Bytes and operations a pass cannot do without.  A product reads its input and writes its
    output once; a Lanczos step reads two vectors and writes one, with the start vector written
    once; an mTPQ step reads one block and writes the next; a CG step also updates its
    solution, residual and direction.  Operations: one multiply-add per matrix element."""
    c = dict(case)
    n, couplings, h, bonds, _, _ = _terms(c)
    rows = sum(math.comb(n, k) for k in range(n + 1)) if c["call"] == "sectors" else _rows(c)
    per = (2 if _complex(c) else 1) * (4 if c.get("prec") == "fp32" else 8)
    # mean matrix elements per row off the diagonal: a bond acts on antiparallel spins in a
    # sector (about half of the rows), on every row in a full basis; a hop on half of the rows
    elems = len(bonds) + (len(couplings) / 2 if not any(h) else 2 * len(couplings) / 3 + n)
    flop = 2 * (elems + 1) * (4 if _complex(c) else 1) * rows
    if c["call"] == "apply":
        return dict(bytes=2 * per * rows * c["nvec"], flops=flop * c["nvec"])
    if c["call"] == "invit":
        return dict(bytes=(2 + 6 * c["steps"]) * 8 * rows, flops=(flop + 10 * rows) * (c["steps"] + 1))
    if c["call"] == "tpq":
        return dict(bytes=(1 + 2 * c["steps"]) * per * rows * c["starts"], flops=flop * c["steps"] * c["starts"])
    steps = c["steps"]
    b = (1 + 3 * steps) * per * rows
    if c["call"] == "refined":  # the Ritz vector from every kept vector, then H x in fp64
        b += steps * per * rows + 3 * 8 * rows
    return dict(bytes=b, flops=(flop + 6 * rows) * (steps + (c["call"] == "refined")))


# ------------------------------------------------------------------------------- 64 bits
def _popcount(x):
    n = torch.zeros_like(x)
    while bool((x != 0).any()):
        n += x & 1
        x = x >> 1
    return n


def _mulhilo(a, x):
    """32-bit words x times the constant a: high and low words (int64 tensors)."""
    p, q = x * (a & 0xFFFF), x * (a >> 16)
    t = p + ((q & 0xFFFF) << 16)
    return (q >> 16) + (t >> 32), t & 0xFFFFFFFF


def _normal(seed, first, count, cplx):
    """Elements first .. first + count - 1 of the seeded start vector: Philox4x32-10 blocks and
    the Box-Muller transform (a block per complex element or per two real ones)."""
    b0, b1 = (first, first + count) if cplx else (first // 2, (first + count + 1) // 2)
    e = torch.arange(b0, b1, device="cuda", dtype=torch.int64)
    w = [e & 0xFFFFFFFF, e >> 32, torch.zeros_like(e), torch.zeros_like(e)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, w[0])
        h1, l1 = _mulhilo(0xCD9E8D57, w[2])
        w = [h1 ^ w[1] ^ k0, l1, h0 ^ w[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    ua = (((w[0] << 21) | (w[1] >> 11)).double() + 0.5) / 2.0**53
    ub = (((w[2] << 21) | (w[3] >> 11)).double() + 0.5) / 2.0**53
    r, t = torch.sqrt(-2.0 * torch.log(ua)), 2.0 * math.pi * ub
    g = torch.stack([r * torch.cos(t), r * torch.sin(t)], dim=1)
    if cplx:
        return torch.view_as_complex(g)
    return g.reshape(-1)[first - 2 * b0: first - 2 * b0 + count]


def _start(seed, rows, nvec, cplx):
    n, step = rows * nvec, 1 << 25
    v = torch.empty(n, device="cuda", dtype=torch.complex128 if cplx else torch.float64)
    for a in range(0, n, step):
        k = min(step, n - a)
        v[a:a + k] = _normal(seed, a, k, cplx)
    return v.view(rows, nvec)


class _SpinH:
    """H on the rows of a spin basis, one gather per distinct flip mask."""

    def __init__(self, c):
        self.n, couplings, h, _, _, _ = _terms(c)
        self.cplx = _complex(c)
        n = self.n
        if "n_up" in c:
            parts = []
            for a in range(0, 1 << n, 1 << 24):
                s = torch.arange(a, min(a + (1 << 24), 1 << n), device="cuda", dtype=torch.int64)
                parts.append(s[_popcount(s) == c["n_up"]].to(torch.int32))
            self.states = torch.cat(parts)
            self.rank = torch.zeros(1 << n, device="cuda", dtype=torch.int32)
            self.rank[self.states.long()] = torch.arange(len(self.states), device="cuda", dtype=torch.int32)
        else:
            self.states = torch.arange(1 << n, device="cuda", dtype=torch.int32)
            self.rank = None
        f = {0: lambda b: 1.0, 1: lambda b: 1j * (1 - 2 * b), 2: lambda b: 2 * b - 1}  # twice S^a, row side
        self.by_mask = {}
        for i, j, J in couplings:
            for a in range(3):
                for b in range(3):
                    if J[a, b]:
                        mask = (1 << i if a < 2 else 0) ^ (1 << j if b < 2 else 0)
                        t = [0.25 * J[a, b] * f[a](q & 1) * f[b](q >> 1) for q in range(4)]
                        had = self.by_mask.setdefault(mask, {}).setdefault((i, j), [0] * 4)
                        for q in range(4):
                            had[q] += t[q]
        for i in range(n):
            for a in range(3):
                if h[a]:
                    t = [-0.5 * h[a] * f[a](q & 1) for q in range(4)]
                    had = self.by_mask.setdefault(1 << i if a < 2 else 0, {}).setdefault((i, i), [0] * 4)
                    for q in range(4):
                        had[q] += t[q]
        self.dim = len(self.states)

    def __call__(self, v):
        w = torch.empty_like(v)
        step = max(1 << 16, (1 << 24) // v.shape[1])
        for a in range(0, self.dim, step):
            s = self.states[a:a + step]
            acc = torch.zeros_like(v[a:a + step])
            for mask, tables in self.by_mask.items():
                coef = 0
                for (i, j), t in tables.items():
                    t = torch.tensor(t, device="cuda", dtype=torch.complex128)
                    t = t if self.cplx else t.real.contiguous()
                    if i == j:
                        coef = coef + t[((s >> i) & 1).long()]
                    else:
                        coef = coef + t[(((s >> i) & 1) | (((s >> j) & 1) << 1)).long()]
                if mask == 0:
                    src = v[a:a + step]
                else:
                    o = s ^ mask
                    src = v.index_select(0, o if self.rank is None else self.rank[o.long()])
                acc.addcmul_(coef.to(v.dtype)[:, None], src)
            w[a:a + step] = acc
        return w

    def observables(self, p):  # p: |x|^2 per row and column
        m = (_popcount(self.states.long()) - 0.5 * self.n).double()
        return torch.zeros_like(p[0]), (m[:, None] * p).sum(0), (m[:, None] ** 2 * p).sum(0)


class _HubbardH:
    """H X = H_dn X + X H_up^T + U n_up n_dn X with X[dn rank][up rank]."""

    def __init__(self, c):
        self.n, _, _, bonds, t, self.U = _terms(c)
        self.cplx = False
        self.up, hu = self._species(c["n_up"], bonds, t)
        self.dn, hd = self._species(c["n_dn"], bonds, t)
        self.hu, self.hd = hu, hd
        self.dim = len(self.up) * len(self.dn)

    def _species(self, k, bonds, t):
        x = np.arange(1 << self.n, dtype=np.int64)
        cnt = sum((x >> i) & 1 for i in range(self.n))
        b = x[cnt == k]
        rank = np.full(1 << self.n, -1, dtype=np.int64)
        rank[b] = np.arange(len(b))
        r, q, w = [], [], []
        for i, j in bonds:
            on = ((b >> i) ^ (b >> j)) & 1 == 1
            between = ((1 << max(i, j)) - 1) & ~((1 << (min(i, j) + 1)) - 1)
            sign = 1 - 2 * (sum((b[on] & between) >> s & 1 for s in range(self.n)) & 1)
            r.append(rank[b[on]])
            q.append(rank[b[on] ^ ((1 << i) | (1 << j))])
            w.append(-t * sign)
        ind = torch.tensor(np.stack([np.concatenate(r), np.concatenate(q)]))
        h = torch.sparse_coo_tensor(ind, torch.tensor(np.concatenate(w).astype(np.float64)), (len(b), len(b)))
        occ = torch.tensor(((b[:, None] >> np.arange(self.n)) & 1).astype(np.float64), device="cuda")
        return occ, h.coalesce().to_sparse_csr().cuda()

    def __call__(self, v):
        x = v.view(len(self.dn), len(self.up))
        w = torch.empty_like(x)
        for a in range(0, len(self.up), 2048):
            w[:, a:a + 2048] = self.hd @ x[:, a:a + 2048].contiguous()
        for a in range(0, len(self.dn), 2048):
            y = x[a:a + 2048]
            w[a:a + 2048] += (self.hu @ y.t().contiguous()).t()
            w[a:a + 2048].addcmul_(self.U * (self.dn[a:a + 2048] @ self.up.t()), y)
        return w.view(-1, 1)

    def observables(self, p):
        p = p.view(len(self.dn), len(self.up))
        d = sum(float((p[a:a + 2048] * (self.dn[a:a + 2048] @ self.up.t())).sum()) for a in range(0, len(self.dn), 2048))
        m = 0.5 * (float(self.up[0].sum()) - float(self.dn[0].sum()))
        one = torch.ones(1, device="cuda", dtype=torch.float64)
        return one * d, one * m * p.sum(), one * m * m * p.sum()


def _h(c):
    return _HubbardH(c) if _terms(c)[3] else _SpinH(c)


def _dot(a, b):
    return float(torch.vdot(a[:, 0], b[:, 0]).real)


def _lanczos(H, v, steps):
    """alpha, beta and the unit Lanczos vectors."""
    alpha, beta, basis = [], [], []
    q, p, b = v / math.sqrt(_dot(v, v)), None, 0.0
    for _ in range(steps):
        basis.append(q)
        u = H(q)
        if p is not None:
            u = u - b * p
        a = _dot(q, u)
        u = u - a * q
        b = math.sqrt(_dot(u, u))
        alpha.append(a)
        beta.append(b)
        if b <= 1e-13 * max(1.0, abs(a)):
            break
        p, q = q, u / b
    t = np.diag(alpha) + np.diag(beta[:-1], 1) + np.diag(beta[:-1], -1)
    ev, y = np.linalg.eigh(t)
    return np.array(alpha), np.array(beta), ev[:1], basis, y[:, 0]


def exact(case, seed):
    c = dict(case)
    if c["call"] == "sectors":
        parts = []
        for k in range(c["n"] + 1):
            H = _SpinH(dict(c, n_up=k))
            parts.append(_lanczos(H, _start(seed + k, H.dim, 1, False), c["steps"])[:3])
        return {k: np.concatenate([p[i] for p in parts]) for i, k in enumerate(("alpha", "beta", "eig"))}
    H = _h(c)
    if c["call"] == "apply":
        # from the vector the call was given: in fp32 the rounded one
        v = _gauss(c, seed, H.dim, c["nvec"])
        if c["prec"] == "fp32":
            v = v.to(torch.complex64 if H.cplx else torch.float32).to(v.dtype)
        return H(v)
    if c["call"] == "invit":
        b = _gauss(c, seed, H.dim, 1)
        shift = 0.1 - _cg_energy(c)
        y, r = b.clone(), b - (H(b) + shift * b)
        p, rr = r.clone(), _dot(r, r)
        for _ in range(c["steps"]):
            if rr <= 1e-24 * _dot(b, b):
                break
            q = H(p) + shift * p
            al = rr / _dot(p, q)
            y, r = y + al * p, r - al * q
            new = _dot(r, r)
            p, rr = r + (new / rr) * p, new
        y = y / math.sqrt(_dot(y, y))
        return dict(x=y[:, 0].contiguous(), e=np.float64(_dot(y, H(y))))
    if c["call"] in ("lanczos", "refined"):
        al, be, eig, basis, y = _lanczos(H, _start(seed, H.dim, 1, H.cplx), c["steps"])
        out = dict(alpha=al, beta=be, eig=eig)
        if c["call"] == "refined":
            x = sum(float(f) * q for f, q in zip(y, basis))
            x = x / math.sqrt(_dot(x, x))
            hx = H(x)
            e = _dot(x, hx)
            out.update(e=np.float64(e), residual=np.float64(torch.linalg.vector_norm(hx - e * x).item()),
                       variance=np.float64(_dot(hx, hx) - e * e))
        return out
    x = _start(seed, H.dim, c["starts"], H.cplx)
    got = {k: np.full((c["steps"], c["starts"]), np.nan) for k in ("u", "h2", "norm", "doublon", "sz", "sz2")}
    group = max(1, min(c["starts"], (1 << 28) // H.dim))  # a few columns at a time
    for g in range(0, c["starts"], group):
        cols = slice(g, g + group)
        y = x[:, cols].contiguous()
        for k in range(c["steps"]):
            n2 = torch.linalg.vector_norm(y, dim=0) ** 2
            hy = H(y)
            u = (y.conj() * hy).real.sum(0) / n2 / H.n
            h2 = torch.linalg.vector_norm(hy, dim=0) ** 2 / n2 / H.n**2
            got["u"][k, cols], got["h2"][k, cols] = u.cpu().numpy(), h2.cpu().numpy()
            if c["obs"] and k % c["obs"] == 0:
                d, m, mm = H.observables((y.conj() * y).real / n2)
                for name, o in (("doublon", d), ("sz", m), ("sz2", mm)):
                    got[name][k, cols] = (o / H.n).cpu().numpy()
            y = (c["l"] * y - hy / H.n) / torch.sqrt(n2)
            nrm = torch.linalg.vector_norm(y, dim=0)
            got["norm"][k, cols] = nrm.cpu().numpy()
            y = y / nrm
    return {k: got[k] for k in list(got)[:6 if c["obs"] else 3]}
