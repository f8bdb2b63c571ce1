"""FP64 same-spin terms as dense sliced products: both tile heights (16 and 96
rows of the same-spin Hamiltonian), unequal and odd string counts, and K-step
lists that leave zero blocks out, against the oracle on sampled rows."""
import numpy as np
import pytest
import torch

import fci_inputs as fi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_1707_04346_gb300 as pkg

    pkg.load()
    return pkg


# 462 x 330 and 792 x 924 strings (16-row tiles), 924 x 924, 715 x 1716 and 1716 x 715 (96-row tiles)
@pytest.mark.parametrize("norb,na,nb", [(11, 5, 4), (12, 5, 6), (12, 6, 6), (13, 4, 6), (13, 6, 4)])
def test_same_spin_products_match_oracle(pkg, oracle_mod, norb, na, nb):
    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    n = ctx.ndet
    c = fi.make_vector(n)
    cd = torch.from_numpy(c).cuda()
    out = torch.empty_like(cd)
    pkg.fci_sigma(ctx, cd, out)
    got = out.cpu().numpy()
    pkg.fci_sigma(ctx, cd, out)
    assert np.array_equal(out.cpu().numpy(), got)  # bit-reproducible
    rng = np.random.default_rng(7)
    rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 1500)])).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c, rows)
    # the FP64 bar: 1e-12 of the largest element
    assert np.abs(got[rows] - ref).max() <= 1e-12 * np.abs(got).max()


# FP32 products: 64-row blocks of C (462 x 330, 20 x 15 strings) and 256-row ones, unequal and
# odd counts; the FP32 bar of the other FP32 kernels
@pytest.mark.parametrize("norb,na,nb", [(6, 3, 2), (11, 5, 4), (12, 6, 6), (13, 4, 6), (13, 7, 6)])
def test_fp32_same_spin_products_match_oracle(pkg, oracle_mod, norb, na, nb):
    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    n = ctx.ndet
    c = fi.make_vector(n).astype(np.float32)
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    pkg.fci_sigma(ctx, torch.from_numpy(c).cuda(), out)
    got = out.double().cpu().numpy()
    rng = np.random.default_rng(8)
    rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 1500)])).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c.astype(np.float64), rows)
    assert np.abs(got[rows] - ref).max() <= 2e-6 * np.abs(got).max()


# one-kernel sigma of small spaces: single electrons, one string per row share, several threads
# per determinant, more strings per row than threads (11; 3,4 has 330, FP32), both precisions
@pytest.mark.parametrize("norb,na,nb", [(2, 1, 1), (5, 4, 1), (7, 2, 5), (9, 5, 4), (12, 1, 2), (13, 11, 1), (11, 3, 4)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_small_space_sigma_matches_oracle(pkg, oracle_mod, norb, na, nb, dtype):
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    n = ctx.ndet
    c = fi.make_vector(n).astype(dtype)
    cd = torch.from_numpy(c).cuda()
    out = torch.full_like(cd, float("nan"))  # overwritten
    pkg.fci_sigma(ctx, cd, out)
    got = out.double().cpu().numpy()
    rows = np.arange(n) if n <= 4000 else np.unique(np.random.default_rng(3).integers(0, n, 2000)).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c.astype(np.float64), rows)
    assert np.abs(got[rows] - ref).max() <= (1e-12 if dtype == np.float64 else 2e-6) * np.abs(ref).max()
    pkg.fci_sigma(ctx, cd, out)
    assert np.array_equal(out.double().cpu().numpy(), got)
