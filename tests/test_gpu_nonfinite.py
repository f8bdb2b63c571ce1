"""A NaN or an infinity in C must not come out as numbers: every element of sigma that the entry
couples to is non-finite, in the FP32 and FP64 tensor-core kernels and in the one-kernel sigma."""
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


# one kernel; fused walk and sigma_3 of small rows; dense products (64-row blocks); per-row FP32
# sigma_3 with 64-row and 256-row blocks
@pytest.mark.parametrize("norb,na,nb", [(8, 4, 4), (10, 5, 5), (11, 6, 5), (12, 6, 6), (13, 7, 6)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_nonfinite_entries_reach_what_they_couple_to(pkg, norb, na, nb, dtype, bad):
    h1, eri = fi.make_integrals(norb, 60)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    n = ctx.ndet
    at = n // 3
    unit = torch.zeros(n, dtype=torch.float64, device="cuda")
    unit[at] = 1.0
    column = torch.empty_like(unit)
    fma = pkg.fci_init(norb, na, nb, h1, eri, pkg.default_options(f64_kernels=1))
    pkg.fci_sigma(fma, unit, column)
    c = torch.from_numpy(fi.make_vector(n)).cuda().to(dtype)
    out = torch.zeros_like(c)
    pkg.fci_sigma(ctx, c, out)
    clean = out.clone()
    c[at] = bad
    pkg.fci_sigma(ctx, c, out)
    assert not torch.isfinite(out[column != 0.0]).any()
    # and nothing of it stays in the context
    c[at] = 0.0
    pkg.fci_sigma(ctx, c, out)
    assert torch.isfinite(out).all() and torch.isfinite(clean).all()
    assert pkg.fci_query(ctx, pkg.fci.FCI_Q_DEVICE_ERROR) == 0
    pkg.fci_free(fma)
    pkg.fci_free(ctx)
