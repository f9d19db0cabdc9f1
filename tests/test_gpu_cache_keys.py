"""Kernel spectra are kept between calls by their geometry.  Two bin sets whose squared
edges differ by less than 1e-6 but lie on either side of an integer hold different
cells: a context that has measured one of them measures the other as a new context
does.  The cells of |r|^2 = 25 change bins between the two sets, which moves the
coefficients by parts in ten; equal sets agree to the order of the sums (FP32 products,
FP64 sums over at most 1024 points: 1e-10 of the largest coefficient)."""
import numpy as np
import pytest

from paper_2210_10206_gb300 import synth

pytestmark = pytest.mark.gpu
BELOW, ABOVE = [1.5, 4.99999999, 7.3], [1.5, 5.00000001, 7.3]  # squared: 24.9999999, 25.0000001


@pytest.fixture(scope="module")
def sbg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_10206_gb300 import build, sbg as s
    build.build()
    return s


def _full(ctx, edges):
    f = synth.lognormal_field(31, (16, 16, 16), 1.0, -2.0, dtype=np.float64)
    return ctx.full(f, edges, lmax3=2)[0]


def _projected(ctx, edges):
    f = synth.lognormal_field(32, (32, 32), 1.0, -2.0, dtype=np.float64)
    return ctx.projected(f, edges, 2, npcf=(3,))[0]


def _slices(ctx, edges):
    f = np.stack([synth.lognormal_field(33 + i, (32, 32), 1.0, -2.0, dtype=np.float64) for i in range(3)])
    return ctx.projected_slices(f, edges, 2, npcf=(3,))[0]


@pytest.mark.parametrize("call", [_full, _projected, _slices])
def test_edges_on_either_side_of_an_integer(sbg, call):
    ctx, fresh = sbg.Context(0), sbg.Context(0)
    first = call(ctx, BELOW)
    again, ref = call(ctx, ABOVE), call(fresh, ABOVE)
    top = np.abs(ref).max()
    assert np.abs(first - ref).max() > 1e-2 * top  # the two sets do differ
    assert np.abs(again - ref).max() <= 1e-10 * top
    ctx.close()
    fresh.close()
