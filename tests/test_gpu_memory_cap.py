"""fci_options.max_device_bytes beside the memory that makes calls faster: what fits without the
kept scratch and the optional tables fits with them."""
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


def held(pkg, ctx):
    return pkg.fci_query(ctx, pkg.fci.FCI_Q_DEVICE_BYTES)


def test_kept_density_scratch_gives_way_to_a_solve(pkg):
    """The scratch that fci_rdm2 leaves with the context is given back when the solver's
    workspace needs the room."""
    norb, na, nb = 8, 4, 4
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    tables = held(pkg, ctx)
    e = pkg.fci_davidson(ctx, 1, 1e-10)
    c = torch.from_numpy(fi.make_vector(ctx.ndet)).cuda()
    g = pkg.fci_rdm2(ctx, c)
    kept = held(pkg, ctx) - tables
    # two bases of 24 vectors, two sets of 8, one vector, and small arrays
    solve = 8 * ctx.ndet * (2 * 24 + 2 * 8 + 1) + (1 << 20)
    pkg.fci_free(ctx)
    assert kept > 0
    ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(max_device_bytes=float(tables + max(kept, solve))))
    for _ in range(2):
        g2 = pkg.fci_rdm2(ctx, c)
        assert np.array_equal(g2[0], g[0]) and np.array_equal(g2[1], g[1])
        assert held(pkg, ctx) == tables + kept
        assert abs(pkg.fci_davidson(ctx, 1, 1e-10) - e).max() < 1e-11
    pkg.fci_free(ctx)


def test_densities_take_less_scratch_where_room_is_short(pkg):
    """fci_rdm2 in smaller chunks of determinants, fci_rdm1 in one row chunk: the same bits of the
    2-RDM, the 1-RDM to rounding, in no more memory than a partial per replacement took."""
    norb, na, nb = 10, 5, 5  # planes of one chunk: 100 MB
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    tables = held(pkg, ctx)
    c = torch.from_numpy(fi.make_vector(ctx.ndet)).cuda()
    g = pkg.fci_rdm2(ctx, c)
    pkg.fci_free(ctx)
    for room in (95e6, 5e6):
        ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(max_device_bytes=tables + room))
        g2 = pkg.fci_rdm2(ctx, c)
        assert np.array_equal(g2[0], g[0]) and np.array_equal(g2[1], g[1])
        pkg.fci_free(ctx)

    norb, na, nb = 13, 6, 5  # many row chunks
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    tables = held(pkg, ctx)
    entries = [pkg.fci_query(ctx, q) for q in (2, 3, 4, 5)]
    c = torch.from_numpy(fi.make_vector(ctx.ndet)).cuda()
    g = pkg.fci_rdm1(ctx, c)
    pkg.fci_free(ctx)
    room = 8.0 * (entries[0] * entries[2] + entries[1] * entries[3] + norb**2) + 4096
    ctx = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(max_device_bytes=tables + room))
    assert np.abs(pkg.fci_rdm1(ctx, c) - g).max() < 1e-13 * (na + nb)
    pkg.fci_free(ctx)
