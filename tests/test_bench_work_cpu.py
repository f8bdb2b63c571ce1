"""The work that bench.py counts for the dense same-spin products: the steps of the same-spin
Hamiltonian that hold a nonzero, as the library keeps them, so that no fraction of a peak
credits products that were left out."""
import math

import numpy as np
import pytest

import bench

PEAKS = {"bf16_tflops": 1887.0, "hbm_gbs": 6700.0}


@pytest.mark.parametrize("norb,ne,rows", [(6, 3, 16), (8, 4, 16), (9, 2, 96), (10, 5, 96), (11, 8, 128), (7, 7, 16), (7, 1, 16)])
def test_kept_elements_against_the_hamiltonian(oracle_mod, norb, ne, rows):
    """The pattern of the one-spin Hamiltonian (nbeta = 0) with dense random integrals."""
    r = np.random.RandomState(3)
    g = r.standard_normal((norb, norb))
    chol = r.standard_normal((norb * norb, norb, norb))
    chol = (chol + chol.transpose(0, 2, 1)).reshape(-1, norb * norb)
    eri = (chol.T @ chol).reshape((norb,) * 4)
    H = oracle_mod.hamiltonian(norb, ne, 0, g + g.T, eri) != 0.0
    ns = H.shape[0]
    assert ns == math.comb(norb, ne)
    np.fill_diagonal(H, False)
    want = 0
    for b in range(0, ns, rows):
        block = H[b:b + rows]
        steps = sum(bool(block[:, k:k + 16].any()) for k in range(0, ns, 16))
        want += len(block) * 16 * max(1, steps)
    assert bench.kept_elements(norb, ne, rows) == want


@pytest.mark.parametrize("name,products", [("sigma1_ss", 21), ("sigma2_ss", 21), ("sigma12_ss32", 6), ("sigma2_ss32", 6)])
def test_products_left_out_are_not_counted(name, products):
    n = 3432
    dense = products * 2.0 * n * n * n * (2 if name == "sigma12_ss32" else 1)
    bound, amount, unit, _, _, _ = bench.kernel_work(name, 14, 7, 7, n * n, 56, 56, n, n, PEAKS)
    # 9 % of the steps of 96-row blocks hold only zeros, 7 % of 128-row blocks'
    assert bound == "tensor" and unit == "TFLOP/s" and 0.85 * dense < amount < 0.95 * dense
