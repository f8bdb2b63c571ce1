"""FP64 and FP32 sigma where one spin has a single string (no or all orbitals occupied), so that a
row or a column of C is one element long, against the oracle on sampled rows."""
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


# full beta: 96-row tiles of the FP64 same-spin products (12870, 12376 strings), the small-space
# kernel; full alpha; the large-space kernels on a space the small-space kernel would take
@pytest.mark.parametrize("norb,na,nb,opts", [
    (16, 8, 16, {}), (17, 6, 17, {}), (12, 6, 12, {}), (16, 16, 8, {}), (16, 6, 16, {"f64_kernels": 3}),
    (16, 16, 6, {"f64_kernels": 3}), (16, 8, 0, {}), (16, 0, 8, {})])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_sigma_with_one_string_of_a_spin(pkg, oracle_mod, norb, na, nb, opts, dtype):
    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(**opts))
    n = ctx.ndet
    c = fi.make_vector(n).astype(dtype)
    out = torch.full((n,), float("nan"), dtype=torch.from_numpy(c).dtype, device="cuda")
    pkg.fci_sigma(ctx, torch.from_numpy(c).cuda(), out)
    got = out.double().cpu().numpy()
    rng = np.random.default_rng(4)
    rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 1000)])).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c.astype(np.float64), rows)
    # the bars of the other sigma tests
    assert np.abs(got[rows] - ref).max() <= (1e-12 if dtype == np.float64 else 2e-6) * np.abs(ref).max()
    pkg.fci_free(ctx)
