"""Densities beside other calls on one context: fci_rdm1 and fci_rdm2 in several host threads while
another thread computes sigma vectors on its own stream.  Every result is bit-reproducible, so each
has to equal the one computed alone."""
import threading

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


# one string space and two; small enough for the one-launch 1-RDM, and larger
@pytest.mark.parametrize("norb,na,nb", [(8, 4, 4), (11, 6, 5), (12, 6, 6)])
def test_densities_beside_sigma_in_other_threads(pkg, norb, na, nb):
    h1, eri = fi.make_integrals(norb, 40)
    ctx = pkg.fci_init(norb, na, nb, h1, eri)
    c = torch.from_numpy(fi.make_vector(ctx.ndet)).cuda()
    out = torch.empty_like(c)
    pkg.fci_sigma(ctx, c, out)
    torch.cuda.synchronize()
    sigma = out.cpu().numpy()
    g1, (d1, d2) = pkg.fci_rdm1(ctx, c), pkg.fci_rdm2(ctx, c)
    wrong, stop = [], threading.Event()

    def guarded(work):
        def body():
            try:
                work()
            except Exception as e:  # seen by the main thread
                wrong.append(repr(e))

        return threading.Thread(target=body)

    def sigmas():
        stream, mine = torch.cuda.Stream(), torch.empty_like(c)
        stream.wait_stream(torch.cuda.default_stream())
        while not stop.is_set():
            pkg.fci_sigma(ctx, c, mine, stream)
            stream.synchronize()
            if not np.array_equal(mine.cpu().numpy(), sigma):
                wrong.append("sigma")

    def rdm1():
        for _ in range(30):
            if not np.array_equal(pkg.fci_rdm1(ctx, c), g1):
                wrong.append("rdm1")

    def rdm2():
        for _ in range(10):
            x1, x2 = pkg.fci_rdm2(ctx, c)
            if not (np.array_equal(x1, d1) and np.array_equal(x2, d2)):
                wrong.append("rdm2")

    s, others = guarded(sigmas), [guarded(w) for w in (rdm1, rdm1, rdm2, rdm2)]
    for t in [s] + others:
        t.start()
    for t in others:
        t.join()
    stop.set()
    s.join()
    assert not wrong, wrong[:5]
    pkg.fci_free(ctx)
