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


def f32_error(pkg, oracle_mod, ctx, space, h1, eri):
    """Largest error of an FP32 sigma on sampled rows, in units of its largest element."""
    c = fi.make_vector(ctx.ndet).astype(np.float32)
    out = torch.empty(ctx.ndet, dtype=torch.float32, device="cuda")
    pkg.fci_sigma(ctx, torch.from_numpy(c).cuda(), out)
    rows = np.unique(np.random.default_rng(5).integers(0, ctx.ndet, 500)).astype(np.int64)
    ref = oracle_mod.sigma_rows(*space, h1, eri, c.astype(np.float64), rows)
    return np.abs(out.double().cpu().numpy()[rows] - ref).max() / np.abs(ref).max()


# one string space (the fused kernel without planes: 8 rows, and 4 at 6435 strings), two spaces (staged)
@pytest.mark.parametrize("space", [(12, 6, 6), (13, 6, 5), (15, 7, 7)])
@pytest.mark.parametrize("f64_kernels", [0, 1])
def test_contexts_without_room_for_the_fp32_planes(pkg, oracle_mod, space, f64_kernels):
    """fci_init leaves the planes of the FP32 same-spin products out where they do not fit, and
    FP32 sigma uses the kernels that need none."""
    if space == (15, 7, 7) and f64_kernels == 0:
        pytest.skip("the same FP32 kernels; 41 million determinants once are enough")
    h1, eri = fi.make_integrals(space[0], 40)
    ctx = pkg.fci_init(*space, h1, eri, pkg.default_options(f64_kernels=f64_kernels))
    full = held(pkg, ctx)
    pkg.fci_free(ctx)
    ctx = pkg.fci_init(*space, h1, eri, pkg.default_options(f64_kernels=f64_kernels, max_device_bytes=float(full - 1)))
    assert held(pkg, ctx) < full
    assert f32_error(pkg, oracle_mod, ctx, space, h1, eri) <= 2e-6  # the bar of the FP32 kernels
    pkg.fci_free(ctx)


@pytest.mark.parametrize("space", [(12, 6, 6), (13, 6, 5)])
def test_fp32_planes_give_way_to_a_solve(pkg, oracle_mod, space):
    """A workspace that does not fit beside the planes of the FP32 products takes their place,
    unless a captured graph may still read them."""
    h1, eri = fi.make_integrals(space[0], 40)
    opts = dict(f64_kernels=1, max_subspace=4, max_iter=2)  # FP64 kernels without planes of their own
    ctx = pkg.fci_init(*space, h1, eri, pkg.default_options(**opts))
    full, n = held(pkg, ctx), ctx.ndet
    pkg.fci_free(ctx)
    solve = 8 * n * (2 * 4 + 2 * 2 + 1)  # the vectors alone
    for captured in (False, True):
        ctx = pkg.fci_init(*space, h1, eri, pkg.default_options(max_device_bytes=float(full + solve - 4096), **opts))
        assert held(pkg, ctx) == full
        if captured:
            c = torch.from_numpy(fi.make_vector(n).astype(np.float32)).cuda()
            out = torch.empty_like(c)
            pkg.fci_sigma(ctx, c, out)
            want = out.clone()
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                pkg.fci_sigma(ctx, c, out)
        with pytest.raises(pkg.FciError) as err:
            pkg.fci_davidson(ctx, 1, 1e-12)
        if captured:
            assert err.value.code == pkg.fci.FCI_ERR_OOM and held(pkg, ctx) == full
            out.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert float((out - want).abs().max()) <= 2e-6 * float(want.abs().max())
        else:
            assert err.value.code == pkg.fci.FCI_ERR_NOCONV and held(pkg, ctx) < full
            assert f32_error(pkg, oracle_mod, ctx, space, h1, eri) <= 2e-6
        pkg.fci_free(ctx)
