"""1-RDM: the one-launch path of small spaces and the pair-list path, on either
side of their limit (20000 determinants), with one and two string spaces, a spin
without electrons, FP32 input and the call without allocation, against the oracle."""
import numpy as np
import pytest
import torch

import fci_inputs as fi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb,na,nb", [(1, 1, 1), (6, 3, 0), (9, 4, 5), (10, 5, 5), (10, 4, 6), (13, 5, 11), (13, 11, 5)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_rdm1_matches_oracle(oracle_mod, norb, na, nb, dtype):
    import paper_1707_04346_gb300 as pkg

    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    c = fi.make_vector(ctx.ndet).astype(dtype)
    cd = torch.from_numpy(c).cuda()
    ref = oracle_mod.rdm1(norb, na, nb, c.astype(np.float64))
    g = pkg.fci_rdm1(ctx, cd)
    assert np.abs(g - ref).max() <= 1e-13 * max(1, na + nb)
    assert np.array_equal(pkg.fci_rdm1(ctx, cd), g)
    assert np.abs(pkg.fci_rdm1_noalloc(ctx, cd) - ref).max() <= 1e-13 * max(1, na + nb)
