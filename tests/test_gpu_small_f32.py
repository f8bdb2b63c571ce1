"""FP32 sigma of small spaces with few strings of one spin, where many threads share a determinant:
adding their parts must not cost more than the roundings of the terms themselves."""
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


# 256 parts (one beta string), 51, 28, 17, 2
@pytest.mark.parametrize("norb,na,nb", [(11, 5, 11), (12, 6, 12), (13, 6, 13), (14, 7, 14), (5, 2, 1), (9, 5, 8), (6, 4, 2), (9, 5, 4)])
def test_parts_of_a_determinant_are_summed_beyond_fp32(pkg, oracle_mod, norb, na, nb):
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    c = fi.make_vector(ctx.ndet).astype(np.float32)
    out = torch.empty(ctx.ndet, dtype=torch.float32, device="cuda")
    pkg.fci_sigma(ctx, torch.from_numpy(c).cuda(), out)
    ref = oracle_mod.sigma(norb, na, nb, h1, eri, c.astype(np.float64))
    # The diagonal dominates: its two FP32 constants, their products' sum and the result are
    # rounded, four roundings of 2^-24 at most each and 2^-24 / sqrt(3) in the mean square, so
    # 1.2 x 2^-24 together; twice that for the couplings' roundings.
    err = np.linalg.norm(out.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 2.4 * 2.0**-24, err
    pkg.fci_free(ctx)
