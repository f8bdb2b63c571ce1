"""FP32 sigma of spaces that the per-row FP32 sigma_3 takes (at least 600 alpha and 769 beta strings)
with four to six K-steps per row, up to 231 orbital pairs and rows of very different length, both
slice counts, rows of C that are zero or on another scale, against the oracle on sampled rows."""
import numpy as np
import pytest
import torch

import fci_inputs as fi

pytestmark = pytest.mark.gpu


# K = 52, 54 (four K-steps, not full), 56, 68, 70 (five), 85 (six); 136 to 231 pairs; 816 to
# 3432 beta strings
@pytest.mark.parametrize("norb,na,nb,ksteps", [(16, 4, 4, 4), (20, 3, 3, 4), (14, 7, 6, 4), (20, 4, 3, 5), (18, 5, 3, 5), (21, 5, 3, 6)])
@pytest.mark.parametrize("splits", [3, 2])
def test_rows_match_oracle(oracle_mod, norb, na, nb, ksteps, splits):
    import paper_1707_04346_gb300 as pkg

    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(f32_splits=splits))
    nsa, nsb = ctx.nstr
    # what the kernel is taken for
    assert nsa >= 600 and nsb >= 769 and -(-pkg.fci_query(ctx, pkg.fci.FCI_Q_NSINGLE_ALPHA) // 16) == ksteps
    n = ctx.ndet
    c = fi.make_vector(n).astype(np.float32).reshape(-1, nsb)
    c[1::7] *= np.float32(2.0**-30)
    c[3::11] = 0.0
    c = c.reshape(-1)
    cd = torch.from_numpy(c).cuda()
    out = torch.empty_like(cd)
    pkg.fci_sigma(ctx, cd, out)
    got = out.cpu().numpy()
    rows = np.unique(np.concatenate([[0, n - 1], np.random.default_rng(9).integers(0, n, 400)])).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c.astype(np.float64), rows)
    # 3 slices: the FP32 bar of the other FP32 kernels; 2 slices (17 bits): its 64-fold
    bar = 2e-6 if splits == 3 else 1.3e-4
    assert np.abs(got[rows] - ref).max() <= bar * np.abs(got).max()
    if max(nsa, nsb) <= 16384:  # beyond, the same-spin terms are summed by FP32 atomics
        pkg.fci_sigma(ctx, cd, out)
        assert np.array_equal(out.cpu().numpy(), got)  # bit-reproducible
    pkg.fci_free(ctx)
