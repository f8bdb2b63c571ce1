"""1-RDM of spaces with few strings of one spin, on either side of the one-launch rule, and pair
lists built by several CTAs (512 strings each, whole and partial), against the oracle."""
import numpy as np
import pytest
import torch

import fci_inputs as fi

pytestmark = pytest.mark.gpu


# one string: (11; 11,5) one launch, (12; 12,6) lists of 924, (15; 15,7) 6435, (13; 6,13) one launch,
# (15; 7,15); few strings: (11; 2,5), (18; 1,4), (14; 4,1) one launch, (13; 2,4), (12; 2,5) lists;
# two spaces either side of the limit (11; 3,3), (9; 4,5); no electrons of a spin; lists of 495, 1287
@pytest.mark.parametrize("norb,na,nb", [
    (11, 11, 5), (12, 12, 6), (15, 15, 7), (13, 6, 13), (15, 7, 15), (11, 2, 5), (18, 1, 4), (14, 4, 1), (13, 2, 4),
    (12, 2, 5), (11, 3, 3), (9, 4, 5), (14, 0, 7), (14, 7, 0), (12, 4, 8), (13, 5, 5), (2, 1, 1)])
def test_rdm1_matches_oracle(oracle_mod, norb, na, nb):
    import paper_1707_04346_gb300 as pkg

    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    c = fi.make_vector(ctx.ndet)
    cd = torch.from_numpy(c).cuda()
    ref = oracle_mod.rdm1(norb, na, nb, c)
    bar = 1e-13 * max(1, na + nb)  # as for the other density tests
    g = pkg.fci_rdm1(ctx, cd)
    assert np.abs(g - ref).max() <= bar
    assert np.array_equal(pkg.fci_rdm1(ctx, cd), g)
    assert np.abs(pkg.fci_rdm1_noalloc(ctx, cd) - ref).max() <= bar
    pkg.fci_free(ctx)
