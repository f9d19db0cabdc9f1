"""Device memory of calls in a context with a budget: each budget below has been enough
for its call since before several groups shared a launch and the FP32 4PCF's entries
were padded to whole thread tiles, and stays enough.  A call in a tight budget may take
other paths than one without (spectra generated anew, fewer fields per slab), which the
parity tests each hold within 1e-5 (split BF16: 1e-4) of the oracle's largest
coefficient: the two results are within twice that of each other."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
FP32, BF16X3 = 0, 1


@pytest.fixture(scope="module")
def sbg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_10206_gb300 import build, sbg as s
    build.build()
    return s


def _edges(n, nb):
    return np.linspace(0.5, 0.4 * n, nb + 1)


@pytest.mark.parametrize("kind,n,nb,order,prec,budget", [
    ("projected", 16, 3, 2, FP32, 71039), ("projected", 16, 3, 2, BF16X3, 105087), ("projected3", 16, 3, 2, FP32, 18815),
    ("projected", 64, 5, 3, FP32, 1748926), ("projected", 64, 20, 2, FP32, 10881269),
    ("projected3", 64, 20, 2, FP32, 1431998), ("slices", 64, 5, 3, FP32, 1748926), ("full", 16, 5, 2, FP32, 1536126),
    ("full", 16, 5, 2, BF16X3, 3424252), ("full3", 16, 5, 2, FP32, 413695), ("odd", 16, 5, 2, FP32, 1477182)])
def test_budget_stays_enough(sbg, kind, n, nb, order, prec, budget):
    rng = np.random.default_rng(n + nb)
    f = rng.random({"full": (n, n, n), "full3": (n, n, n), "odd": (n, n, n), "slices": (5, n, n)}.get(kind, (n, n)))
    calls = {"projected": lambda c: c.projected(f, _edges(n, nb), order, prec=prec),
             "projected3": lambda c: c.projected(f, _edges(n, nb), order, npcf=(3,)),
             "slices": lambda c: c.projected_slices(f, _edges(n, nb), order),
             "full": lambda c: c.full(f, _edges(n, nb), lmax3=order, lmax4=order, prec=prec),
             "full3": lambda c: c.full(f, _edges(n, nb), lmax3=order),
             "odd": lambda c: (None, c.full_odd(f, _edges(n, nb), order))}
    tight, free = sbg.Context(0, budget=budget), sbg.Context(0)
    for a, b in zip(calls[kind](tight), calls[kind](free)):
        if b is not None:
            assert np.abs(a - b).max() <= 2 * (1e-4 if prec else 1e-5) * np.abs(b).max()
    tight.close()
    free.close()
