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
