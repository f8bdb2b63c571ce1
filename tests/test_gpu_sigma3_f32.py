"""FP32 sigma_3 with the sigma row in shared memory, where its tiles can go wrong:
one K-step and a partly filled one, every padding of the pair count, rows shorter
than a tile and one string past a tile, both slice counts, a row of C that is zero
or far smaller than its neighbours."""
from math import comb

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


# replacements K = 15 (one K-step, not full), 20, 27, 33, 48 and 45 (full and not full),
# rows of 1365, 462, 165, 1716, 715 and 715 strings
@pytest.mark.parametrize("norb,na,nb,splits", [
    (15, 1, 4, 3), (11, 2, 5, 3), (11, 3, 8, 2), (13, 3, 7, 3), (13, 6, 4, 3), (13, 9, 4, 2),
    # at least 600 x 769 strings: 715 x 1287 (K = 40, 45), 792 x 792 (K = 40), 1001 x 1001 (K = 44
    # and 50 targets a string), 816 x 816 (K = 48, 171 pairs)
    (13, 4, 5, 3), (13, 9, 8, 2), (12, 5, 5, 3), (14, 4, 10, 2), (18, 3, 3, 3),
])
def test_rows_match_oracle(pkg, oracle_mod, norb, na, nb, splits):
    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(f32_splits=splits))
    n, nsb = ctx.ndet, comb(norb, nb)
    c = fi.make_vector(n).astype(np.float32).reshape(-1, nsb)
    c[1::7] *= np.float32(2.0 ** -30)  # rows on other scales
    c[3::11] = 0.0
    c = c.reshape(-1)
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    cd = torch.from_numpy(c).cuda()
    pkg.fci_sigma(ctx, cd, out)
    got = out.double().cpu().numpy()
    rng = np.random.default_rng(9)
    rows = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 1500)])).astype(np.int64)
    ref = oracle_mod.sigma_rows(norb, na, nb, h1, eri, c.astype(np.float64), rows)
    # 3 slices: the FP32 bar of the other FP32 kernels; 2 slices (17 bits): its 64-fold
    bar = 2e-6 if splits == 3 else 1.3e-4
    assert np.abs(got[rows] - ref).max() <= bar * np.abs(got).max()
    pkg.fci_sigma(ctx, cd, out)
    assert np.array_equal(out.double().cpu().numpy(), got)  # bit-reproducible
