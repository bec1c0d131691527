"""Every launch shape of the two-pass Hubbard path against the oracle: 1, 2 and 4 pieces a lane of the
down-spin pass, 1, 2 and 4 rows a tile of the up-spin pass, rows that start on 16 bytes and not."""
import numpy as np
import pytest

import oracle
import workloads as wl

torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_1703_03637_gb300")

pytestmark = pytest.mark.gpu

PRECS = [(hp.FP64, 1e-12), (hp.FP32, 2e-5)]  # of the largest element, as for the other products
SHAPES = [(p, k) for p in (1, 2, 4) for k in (1, 2, 4)]


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("n,nu,nd", [
    (12, 6, 3),  # rows of 924, a multiple of 16 bytes, four stripes of four fp64 pieces, 220 down rows
    (15, 7, 1),  # rows of 6,435: odd, so element by element, and a last tile of 3 rows in 4
    (7, 3, 2),   # rows of 35, shorter than any stripe
])
def test_every_shape(n, nu, nd):
    spec = wl.hubbard(n, wl.ring_bonds(n) + wl.ring_bonds(n, 2), 1.0, 8.0).with_basis(wl.BASIS_NUMBER, nu, nd)
    m = hp.Model.from_spec(spec)
    v = wl.gaussian_vector(13 * n + nd, m.dim)[:, 0]
    ref = oracle.apply_H(spec, v).real
    a, b = oracle.lanczos(spec, v, 2)
    for prec, tol in PRECS:
        for offset in (0, 1):
            buf = torch.zeros(2, m.dim + 1, device="cuda", dtype=m.dtype(prec))
            x, w = buf[0, offset:offset + m.dim], buf[1, offset:offset + m.dim]
            x.copy_(torch.as_tensor(v))
            for pieces, rows in SHAPES:
                m.set_hubbard_shape(prec, pieces, rows)
                w.fill_(float("nan"))
                m.apply_H(x, w)
                assert _rel(w.cpu().numpy(), ref) < tol, (prec, offset, pieces, rows)
        for pieces, rows in SHAPES:
            m.set_hubbard_shape(prec, pieces, rows)
            r = m.lanczos(2, prec=prec, v0=torch.as_tensor(v))
            assert _rel(r["alpha"], a) < tol and _rel(r["beta"], b) < tol, (prec, pieces, rows)


@pytest.mark.parametrize("nd", [1, 2])
def test_one_long_row_a_tile(nd):
    """17 sites, 8 up: rows of 24,310, one a tile in fp64 (8-byte table) and two in fp32 by default;
    with 2 down, 136 down rows give the down-spin pass its two pieces a lane by default."""
    spec = wl.hubbard_ring(17, 1.0, 8.0).with_basis(wl.BASIS_NUMBER, 8, nd)
    m = hp.Model.from_spec(spec)
    v = wl.gaussian_vector(17 + nd, m.dim)[:, 0]
    ref = oracle.apply_H(spec, v).real
    a, b = oracle.lanczos(spec, v, 2)
    for prec, tol in PRECS:
        w = m.apply_H(torch.as_tensor(v).to(device="cuda", dtype=m.dtype(prec)))
        assert _rel(w.cpu().numpy(), ref) < tol
        r = m.lanczos(2, prec=prec, v0=torch.as_tensor(v))
        assert _rel(r["alpha"], a) < tol and _rel(r["beta"], b) < tol


def test_shape_arguments():
    m = hp.Model.from_spec(wl.hubbard_ring(6).with_basis(wl.BASIS_NUMBER, 3, 3))
    for bad in ((3, 1), (1, 3), (-1, 1), (8, 1)):
        with pytest.raises(hp.LibraryError) as e:
            m.set_hubbard_shape(hp.FP64, *bad)
        assert e.value.code == -1
    with pytest.raises(hp.LibraryError) as e:
        hp.Model.from_spec(wl.heisenberg_ring(6)).set_hubbard_shape(hp.FP64, 1, 1)
    assert "two-pass" in str(e.value)
    m.set_hubbard_shape(hp.FP64, 0, 0)
