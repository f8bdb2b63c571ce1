"""fci_rdm2's Gram tiles where they can go wrong: blocks of one padded row, of one
tile, of two column tiles with whole planes (13 and 15 orbitals), of two row tiles
with planes copied by tile (16: S only; 17: both blocks), unequal spins, fewer
determinants than one accumulator group, a vector of equal elements (largest digits)
and partial groups at chunk ends."""
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


@pytest.mark.parametrize("norb,na,nb", [(1, 1, 0), (2, 2, 1), (3, 1, 2), (11, 1, 2), (13, 2, 1), (14, 1, 1), (15, 1, 2),
                                        (16, 2, 1), (17, 1, 2)])
def test_tiles_match_oracle(pkg, oracle_mod, norb, na, nb):
    h1, eri = fi.make_integrals(norb, 30)
    n = oracle_mod.ndet(norb, na, nb)
    c = fi.make_vector(n)
    c /= np.linalg.norm(c)
    ref2, ref1 = oracle_mod.rdm2(norb, na, nb, c), oracle_mod.rdm1(norb, na, nb, c)
    got = []
    for chunk in (0.0, 1.0):  # the default and the smallest chunk, one accumulator group
        ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(rdm2_chunk_bytes=chunk))
        got.append(pkg.fci_rdm2(ctx, torch.from_numpy(c).cuda()))
        e = np.full(n, -1.0)  # every digit of c is its largest: exact integers throughout
        g1, g2 = pkg.fci_rdm2(ctx, torch.from_numpy(e).cuda())
        assert np.array_equal(g2, oracle_mod.rdm2(norb, na, nb, e))
        assert np.array_equal(g1, oracle_mod.rdm1(norb, na, nb, e))
        pkg.fci_free(ctx)
    for g1, g2 in got:
        # the bar of the other 2-RDM comparisons
        assert np.abs(g2 - ref2).max() <= 1e-12
        assert np.abs(g1 - ref1).max() <= 1e-12
        assert np.array_equal(g2, got[0][1]) and np.array_equal(g1, got[0][0])
