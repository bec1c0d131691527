"""Roundings that the library's results are allowed: each operation of the method rounds once, on
inputs whose exact results are known."""
import math

import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_1703_03637_gb300")

pytestmark = pytest.mark.gpu


# ----------------------------------------------------------------------------- one-cluster Lanczos scalars
def test_one_cluster_square_root_and_reciprocal():
    """Two spins in fields (h_i, 0, z_i) from the all-down state: |C_1|^2 = (h_1^2 + h_2^2) / 4 and
    <C_1, H C_1> are exact, so beta_0 is the correctly rounded square root and alpha_1 the
    product with the correctly rounded reciprocal, bit for bit."""
    for h1 in range(1, 17):
        for h2 in range(1, h1 + 1):
            spec = wl.ModelSpec(kind=wl.SPIN, n_sites=2, couplings=[], fields=[(0, (float(h1), 0.0, 2.0)), (1, (float(h2), 0.0, 1.0))],
                                name="two_spins")
            m = hp.Model.from_spec(spec)
            r = m.lanczos(2, v0=torch.tensor([1.0, 0.0, 0.0, 0.0], dtype=torch.float64))
            ps = (h1 * h1 + h2 * h2) / 4
            xs = (-0.5 * h1 * h1 + 0.5 * h2 * h2) / 4  # the two flipped states' diagonals are -1/2 and 1/2
            b = math.sqrt(ps)
            s = 1.0 / b
            assert r["alpha"][0] == 1.5 and r["beta"][0] == b, (h1, h2)
            assert r["alpha"][1] == xs * s * s, (h1, h2)


# ----------------------------------------------------------------------------- inverse iteration
def _product_state(h, excited):
    """Amplitudes of the product eigenstate of -sum h_i . S_i with spin `excited` (or none) flipped
    against its field, in long double; bit i of the index is spin i up."""
    L = np.longdouble
    v = np.ones(1, L)
    for i, (hx, _, hz) in enumerate(h):
        g = np.array([L(hx), np.sqrt(L(hx) ** 2 + L(hz) ** 2) + L(hz)], L)  # down, up
        g /= np.sqrt((g * g).sum())
        if i == excited:
            g = np.array([-g[1], g[0]], L)
        v = np.outer(g, v).ravel()
    return v


def _fields_times(h, x):
    L = np.longdouble
    out = np.zeros_like(x)
    for i, (hx, _, hz) in enumerate(h):
        a, o = x.reshape(-1, 2, 1 << i), out.reshape(-1, 2, 1 << i)
        o[:, 0] += L(hz) / 2 * a[:, 0] - L(hx) / 2 * a[:, 1]
        o[:, 1] -= L(hx) / 2 * a[:, 0] + L(hz) / 2 * a[:, 1]
    return out


@pytest.mark.parametrize("k", range(4))
def test_inverse_iteration_step_next_to_an_eigenvalue(k):
    """One CG step from b = e + zeta g, A e = e and A g = lambda g with lambda = 2^-30 of the size of
    H: the direction is zeta g, so the step length is 1 / <g, A g> and the iterate shows it.
    Each of the products p_i (A p)_i carries a rounding of |E| p_i, independent of the others:
    an error of 2^-53 |E| (sum g^4)^(1/2) / lambda of the step; 16 times that is allowed.  The
    difference of the sums <p, H p> and c <p, p> would err by 2^-53 |E| / lambda instead, 400 times
    the root here."""
    n, lam, zeta = 16, 2.0 ** -30 * (1 + k / 16), 2.0 ** -13
    rng = np.random.default_rng(4)
    ang = rng.uniform(-10, 10, n) * np.pi / 180
    mag = np.concatenate([[1 - lam], rng.uniform(1.0, 1.5, n - 1)])
    h = [(float(m * np.cos(a)), 0.0, float(m * np.sin(a))) for m, a in zip(mag, ang)]
    L = np.longdouble
    size = [np.sqrt(L(x) ** 2 + L(z) ** 2) for x, _, z in h]
    e0 = -sum(size) / 2
    g, e = _product_state(h, None), _product_state(h, 0)
    b = (e + L(zeta) * g).astype(np.float64)
    energy = float(e0 + size[0])  # c = 1 - energy puts e at one
    c = L(1.0 - energy)
    r = b - (_fields_times(h, b.astype(L)) + c * b)
    step = (r @ r) / (r @ (_fields_times(h, r) + c * r))
    m = hp.Model.from_spec(wl.ModelSpec(kind=wl.SPIN, n_sites=n, couplings=[], fields=list(enumerate(h)), name="fields"))
    x = torch.as_tensor(b).cuda()
    m.inverse_iteration(x, energy, shift=1.0, outer=1, max_cg=1)
    x = x.cpu().numpy().astype(L)
    t = (g @ x) / (e @ x)  # x ~ b + step r
    got = (t * (e @ b) - g @ b) / (g @ r - t * (e @ r))
    s4 = float(np.sqrt((g ** 4).sum()))
    assert abs(got / step - 1) <= 16 * 2.0 ** -53 * abs(float(e0)) * s4 / lam


def test_inverse_iteration_iterate_in_extended_precision():
    """Six CG steps on a split-row sector (12,870 rows) against the same recurrence in long double.
    The products' input is quantised at 2^-57 of its largest element, at most 2^-53 of the typical
    one here, so every operation errs by about one fp64 rounding; 16 of them per element, in the
    root mean square over the vector, cover the six steps' four operations each (24^(1/2) = 5) with
    the conditioning of the recurrence."""
    n, steps, c = 16, 6, 0.1 + 0.4461935 * 16
    spec = wl.heisenberg_ring(n).with_basis(wl.BASIS_SZ, n // 2)
    m = hp.Model.from_spec(spec)
    states = m.basis_states().cpu().numpy()
    rank = np.zeros(1 << n, dtype=np.int64)
    rank[states] = np.arange(len(states))
    L = np.longdouble
    diag, pairs = np.zeros(len(states), L), []
    for i in range(n):
        j = (i + 1) % n
        anti = ((states >> i) ^ (states >> j)) & 1
        diag += np.where(anti, L(-0.25), L(0.25))
        rows = np.nonzero(anti)[0]
        pairs.append((rows, rank[states[rows] ^ (1 << i) ^ (1 << j)]))

    def product(x):
        out = (diag + L(1.0 - (1.0 - c))) * x
        for rows, partner in pairs:
            out[rows] += x[partner] / 2
        return out

    b = np.random.default_rng(11).standard_normal(len(states))
    y = b.astype(L)
    r = y - product(y)
    p = r.copy()
    for _ in range(steps):
        q = product(p)
        rr = r @ r
        al = rr / (p @ q)
        y = y + al * p
        r = r - al * q
        p = r + (r @ r) / rr * p
    x = torch.as_tensor(b).cuda()
    m.inverse_iteration(x, 1.0 - c, shift=1.0, outer=1, max_cg=steps)
    err = x.cpu().numpy().astype(L) - y / np.sqrt(y @ y)
    assert float(np.sqrt(err @ err)) <= 16 * 2.0 ** -53


# ----------------------------------------------------------------------------- infinities in blocks of vectors
@pytest.mark.parametrize("n,nvec,complex_", [(19, 16, False), (16, 64, False), (17, 16, True), (16, 64, True)])
def test_infinity_stays_in_coupled_rows(n, nvec, complex_):
    """An infinite amplitude in a single-precision block reaches the rows with a matrix element to
    its own and no others: all others are bit for bit those of the block with a zero there."""
    D = 0.3 if complex_ else 0.0
    J = np.array([[1.0, D, 0.0], [-D, 1.0, 0.0], [0.0, 0.0, 0.7]])  # an exchange: zero on parallel spins
    m = hp.Model.from_spec(wl.ModelSpec(kind=wl.SPIN, n_sites=n, couplings=[(i, (i + 1) % n, J) for i in range(n)],
                                        name="exchange_ring"))
    assert m.is_complex == complex_
    g = torch.Generator().manual_seed(3)
    v = torch.randn((m.dim, nvec), dtype=m.dtype(hp.FP32), generator=g).cuda()
    row = int("0110100111010010110"[:n], 2)
    coupled = [row] + [row ^ (1 << i) ^ (1 << ((i + 1) % n)) for i in range(n) if (row >> i ^ row >> ((i + 1) % n)) & 1]
    v[row, 1] = 0
    clean = m.apply_H(v)
    v[row, 1] = float("inf")
    w = m.apply_H(v)
    rest = torch.ones(m.dim, dtype=torch.bool, device="cuda")
    rest[coupled] = False
    assert torch.equal(torch.view_as_real(w[rest]) if complex_ else w[rest], torch.view_as_real(clean[rest]) if complex_ else clean[rest])
    assert not torch.isfinite(w[coupled, 1]).any()


# ----------------------------------------------------------------------------- fp64 blocks of vectors
@pytest.mark.parametrize("nvec", [16, 128])
@pytest.mark.parametrize("mk,n,hx", [(wl.heisenberg_ring, 18, 0.0), (wl.j1j2_ring, 18, 0.0), (wl.heisenberg_ring, 18, 1e-3)],
                         ids=["one-class", "two-classes", "weak-field"])
def test_block_products_round_twice(mk, n, hx, nvec):
    """fp64 blocks, most couplings powers of two: besides the quantised copy (2^-57 of the
    column's largest, well below a rounding) an element is rounded when its exchange sum becomes fp64
    and when the diagonal joins.  A rounding's root mean square is 0.42 2^-53 of its value, and the
    exchange part is no larger than 1.1 times the whole here: (1 + 1.1^2)^(1/2) 0.42 < 0.63."""
    spec = mk(n)
    if hx:
        spec.fields = [(i, (hx, 0.0, 0.0)) for i in range(n)]
    m = hp.Model.from_spec(spec)
    L = np.longdouble
    states = np.arange(m.dim)
    g = torch.Generator().manual_seed(9)
    v = torch.randn((m.dim, nvec), dtype=torch.float64, generator=g)
    w = m.apply_H(v.cuda()).cpu().numpy()
    for c in (0, nvec - 1):
        x = v[:, c].numpy().astype(L)
        off, diag = np.zeros(m.dim, L), np.zeros(m.dim, L)
        for i, j, J in spec.couplings:
            anti = ((states >> i) ^ (states >> j)) & 1
            diag += L(J[2, 2]) * np.where(anti, L(-0.25), L(0.25))
            rows = np.nonzero(anti)[0]
            off[rows] += L(J[0, 0]) / 2 * x[states[rows] ^ (1 << i) ^ (1 << j)]
        for i, h in spec.fields:
            off -= L(h[0]) / 2 * x[states ^ (1 << i)]
        ref = off + diag * x
        assert float((off @ off) / (ref @ ref)) < 1.1 ** 2
        err = w[:, c].astype(L) - ref
        assert float(np.sqrt((err @ err) / (ref @ ref))) <= 0.63 * 2.0 ** -53


@pytest.mark.parametrize("mk,nvec", [(lambda: wl.kitaev_honeycomb(4, 2), 64), (lambda: wl.kitaev_honeycomb(4, 2, h=0.3), 32),
                                     (lambda: wl.random_spin_model(16, 12, seed=21), 64)],
                         ids=["kitaev", "kitaev-strong-field", "random"])
def test_block_products_keep_zeros(mk, nvec):
    """fp64 blocks of basis vectors: an element without a matrix element to its column's basis vector is
    zero, and so is a zero column, also where the coefficients' products are rounded."""
    spec = mk()
    m = hp.Model.from_spec(spec)
    rng = np.random.default_rng(12)
    rows = rng.integers(0, m.dim, nvec - 1)
    v = np.zeros((m.dim, nvec), dtype=np.complex128 if m.is_complex else np.float64)
    v[rows, np.arange(nvec - 1)] = rng.uniform(0.5, 2, nvec - 1)
    w = m.apply_H(torch.as_tensor(v).cuda()).cpu().numpy()
    assert not w[:, -1].any()
    for c in range(0, nvec - 1, 7):
        allowed = {rows[c]} | {rows[c] ^ (1 << i) ^ (1 << j) for i, j, _ in spec.couplings}
        allowed |= {rows[c] ^ (1 << i) for i in range(spec.n_sites)}  # fields, and S^z times S^x or S^y
        assert set(np.nonzero(w[:, c])[0].tolist()) <= allowed
