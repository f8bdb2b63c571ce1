"""Davidson of one spin parity on spaces beyond the one-kernel sigma, where sigma_1 is formed from
sigma_2 by the transpose-add: FP64 next to the sliced sigma_3 (16-row and 96-row tiles of the dense
products) and FP32 (64-row and 256-row blocks of C).  The vectors have the parity and are eigenvectors
of the full Hamiltonian, and the energies are those of a solve with the FP64 multiply-add kernels,
which know no parity."""
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


@pytest.mark.parametrize("norb,ne", [(10, 5), (11, 5), (12, 6), (13, 6)])
@pytest.mark.parametrize("opts", [{}, {"precision": 1}, {"precision": 1, "basis_f32": 1}], ids=["fp64", "mixed", "f32basis"])
def test_parity_solutions_are_eigenvectors(pkg, norb, ne, opts):
    if norb == 13 and "basis_f32" in opts:
        pytest.skip("the same sigma kernels as in the mixed solve")
    h1, eri = fi.make_integrals(norb, 60)
    tol = 1e-9  # residuals below 3.2e-5
    for par in (1, -1):
        full = pkg.fci_init(norb, ne, ne, h1, eri, pkg.default_options(spin_parity=par, f64_kernels=1, max_iter=1000))
        ns = full.nstr[0]
        ctx = pkg.fci_init(norb, ne, ne, h1, eri, pkg.default_options(spin_parity=par, max_iter=1000, **opts))
        x = torch.empty((1, ctx.ndet), dtype=torch.float64, device="cuda")
        e = pkg.fci_davidson(ctx, 1, tol, vecs=x)
        c = x[0].reshape(ns, ns)
        assert float((c - par * c.T).abs().max()) < 1e-12
        hx = torch.empty_like(x[0])
        pkg.fci_sigma(full, x[0], hx)
        # the solver's own bar on the residual, twice for the FP32 basis' rounding
        assert float((hx - e[0] * x[0]).norm()) < 2 * np.sqrt(tol)
        assert abs(float(x[0] @ hx) - e[0]) < 1e-8
        assert abs(pkg.fci_davidson(full, 1, tol)[0] - e[0]) < 1e-8
        pkg.fci_free(ctx)
        pkg.fci_free(full)
