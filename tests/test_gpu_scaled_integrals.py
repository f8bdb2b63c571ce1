"""Integrals far from one: powers of two put the Hamiltonian, and with it the projected matrix of
the solvers and the FP32 operands, near and past FP32's range.  Scaling by a power of two is exact,
so the results are those of the unscaled integrals, scaled."""
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


# the energy bar is far above (1e-7)^2 of the spread, what residuals of 1e-7 of the scale leave
@pytest.mark.parametrize("power", [-20, 0, 20, 122, 130, 300])
def test_solves_of_scaled_integrals(pkg, oracle_mod, power):
    norb, na, nb = 6, 3, 3
    h1, eri = fi.make_integrals(norb, 20)
    s = 2.0**power
    w = np.linalg.eigvalsh(oracle_mod.hamiltonian(norb, na, nb, h1, eri))
    ctx = pkg.fci_init(norb, na, nb, h1 * s, eri * s)
    e = pkg.fci_davidson(ctx, 2, (1e-7 * s) ** 2) / s
    assert np.abs(e - w[:2]).max() < 1e-10
    pkg.fci_free(ctx)
    if power > 60:  # the batch pads its projected matrices with 1e30
        return
    h4, eri4 = fi.make_integrals(4, 10)
    batch = pkg.fci_batch_init([(norb, na, nb, h1 * s, eri * s), (4, 2, 2, h4 * s, eri4 * s)])
    e = pkg.fci_batch_davidson(batch, 2, (1e-7 * s) ** 2)
    assert np.abs(e[0] / s - w[:2]).max() < 1e-9
    pkg.fci_batch_free(batch)
