"""The launch counts that results report, kernel by kernel, below and above the size up to which one
kernel scans and quantises an fp64 vector."""
import gc

import pytest

import workloads as wl

torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_1703_03637_gb300")

pytestmark = pytest.mark.gpu

MODELS = [
    # two-pass Hubbard and split-row sector; rows; kernels of one scan and quantisation
    (lambda: wl.hubbard_tilted8().with_basis(wl.BASIS_NUMBER, 4, 4), 4900, 1),
    (lambda: wl.hubbard_ring(10).with_basis(wl.BASIS_NUMBER, 5, 4), 52920, 2),
    (lambda: wl.heisenberg_ring(16).with_basis(wl.BASIS_SZ, 8), 12870, 1),
    (lambda: wl.heisenberg_ring(18).with_basis(wl.BASIS_SZ, 9), 48620, 2),
]


@pytest.mark.parametrize("mk,rows,quant", MODELS, ids=["hubbard-short", "hubbard", "sector-short", "sector"])
def test_launch_counts(mk, rows, quant):
    m = hp.Model.from_spec(mk())
    assert m.dim == rows
    if m.kind == hp.SPIN_HALF and rows <= 32768:  # (fp64 Lanczos runs in one cluster there)
        r = m.lanczos(3, refine=True, keep_basis=1)
        tail = 1 + 3 + (quant + 2)  # Ritz vector; product, energy, residual, finaliser
    else:
        r, tail = m.lanczos(3), 0
    # start vector, its norm and finaliser; per step the two passes, pass 2 and two finalisers, the
    # copy in the first step only; the eigensolver
    assert r["launches"] == 1 + 2 + quant + 3 * (2 + 3) + 1 + tail
    r = m.lanczos(3, prec=hp.FP32)
    assert r["launches"] == 1 + 2 + 3 * (2 + 3) + 1
    x = m.random_vector(5)[:, 0].contiguous()
    r = m.inverse_iteration(x, -100.0, shift=0.1, outer=1, max_cg=3, cg_tol=1e-30)
    assert r["cg_steps"] == 3
    # start: product, residual, finaliser; per iteration the product on a copy (scanned in the first
    # only), step, residual, test, direction; norm in three; Rayleigh quotient: product and four
    assert r["launches"] == (quant + 2 + 2) + (quant + 2 + 4) + 2 * (1 + 2 + 4) + 3 + (quant + 2 + 4)
    if m.kind == hp.HUBBARD:
        r = m.tpq(1, 3, l=8.0)
        assert r["launches"] == 1 + 2 + 3 * (quant + 2 + 1)


def test_high_part_tables_are_shared():
    """Pass H's tables (12 bytes for each of 2^22 high parts here) belong to the sector: neither the
    second precision nor another split of the row pass adds a copy."""
    def used():
        gc.collect()  # models of earlier tests
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free

    hp.Model.from_spec(wl.heisenberg_ring(18).with_basis(wl.BASIS_SZ, 2))  # the context's own memory
    high = 12 << 22
    before = used()
    m = hp.Model.from_spec(wl.heisenberg_ring(34).with_basis(wl.BASIS_SZ, 4))
    built = used()
    assert high <= built - before < 2 * high
    m.set_sector_split(hp.FP64, 15, 2)
    m.set_sector_split(hp.FP32, 16, 1)
    assert used() - built < high
