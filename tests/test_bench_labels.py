"""The kernel names that bench.py writes beside its H v times follow the library's dispatch: tile passes
for a power of two of vectors, rows of 64 bytes or more and two 64 KB tiles for each of 152 SMs."""
import types

import pytest

import bench
import paper_1703_03637_gb300 as hp
import workloads as wl


@pytest.mark.parametrize("n,nvec,complex_,prec,kernel", [
    (16, 64, True, hp.FP32, "k_hv_tile"),    # 512 tiles
    (16, 32, True, hp.FP32, "k_hv_batch"),   # 256 tiles: too few
    (16, 32, True, hp.FP64, "k_maxexp_cols + k_hv_tile"),
    (14, 64, True, hp.FP32, "k_hv_batch"),
    (20, 4, True, hp.FP32, "k_hv_spin"),     # rows of 32 bytes
    (20, 8, True, hp.FP32, "k_hv_tile"),
    (24, 4, True, hp.FP64, "k_maxexp_cols + k_hv_tile"),
    (20, 24, True, hp.FP32, "k_hv_spin"),    # not a power of two
])
def test_block_kernels(n, nvec, complex_, prec, kernel):
    spec = wl.ModelSpec(kind=wl.SPIN, n_sites=n)
    m = types.SimpleNamespace(is_complex=complex_)
    assert bench.hv_group_name(spec, m, prec, nvec, "mTPQ step", sms=152) == f"{kernel} (mTPQ step)"
    sector = spec.with_basis(wl.BASIS_SZ, n // 2)
    assert bench.hv_group_name(sector, m, prec, nvec, "product", sms=152) == "k_hv_spin (product)"
