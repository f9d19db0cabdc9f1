"""GPU parity of the FP32 4PCF contraction at the edges of its tiling: one row and
one column, columns past one group of 64, tiles of 4 and of 8 columns per thread,
row groups that do not fill a tile, the imaginary-part (odd) mode, complex T and
slabs of fields, normalised and not, on grids whose x-splits end within a span.
Tolerance (as for every FP32 output): max |zeta_gpu - zeta_oracle| <= 1e-5 max
|zeta_oracle|."""
import numpy as np
import pytest

from oracle import cpp
from oracle import sarabande_oracle as O
from paper_2210_10206_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ctx():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_10206_gb300 import build, sbg
    build.build()
    c = sbg.Context(0)
    yield c
    c.close()


def _err(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("n,nb,lmax", [(8, 1, 0), (8, 3, 1), (16, 5, 4), (16, 7, 3), (16, 20, 3), (32, 2, 5)])
def test_full(ctx, n, nb, lmax):
    f = synth.lognormal_field(700 + nb, (n, n, n), 1.0, -2.0, dtype=np.float64)
    edges = np.linspace(0.5, 0.46 * n, nb + 1)
    d, _ = O.preprocess(f)
    _, z4 = ctx.full(f, edges, lmax4=lmax)
    assert _err(z4, cpp.zeta4_full(d, edges, lmax)) < TOL


@pytest.mark.parametrize("n,nb,lmax", [(8, 3, 1), (16, 9, 3), (16, 4, 4)])
def test_full_odd(ctx, n, nb, lmax):
    f = synth.lognormal_field(720 + nb, (n, n, n), 1.0, -2.0, dtype=np.float64)
    edges = np.linspace(0.5, 0.46 * n, nb + 1)
    d, _ = O.preprocess(f)
    assert _err(ctx.full_odd(f, edges, lmax), cpp.zeta4_full(d, edges, lmax, odd=True)) < TOL


@pytest.mark.parametrize("n,nb,mmax", [(8, 1, 0), (16, 20, 3), (64, 13, 2), (32, 5, 10)])
def test_projected(ctx, n, nb, mmax):
    f = synth.lognormal_field(740 + nb, (n, n), 1.0, -2.0, dtype=np.float64)
    edges = np.linspace(0.5, 0.46 * n, nb + 1)
    d, _ = O.preprocess(f)
    _, z4 = ctx.projected(f, edges, mmax, npcf=(4,))
    r4 = O.zeta4_projected(d, edges, mmax)
    assert _err(z4[..., 0] + 1j * z4[..., 1], r4) < TOL


def test_slab(ctx):
    n, nb, mmax = 16, 6, 3
    cube = np.stack([synth.lognormal_field(760 + i, (n, n), 1.0, -2.0, dtype=np.float64) for i in range(7)])
    edges = np.linspace(0.5, 7.0, nb + 1)
    _, z4 = ctx.projected_slices(cube, edges, mmax, npcf=(4,))
    for i in range(len(cube)):
        d, _ = O.preprocess(cube[i])
        assert _err(z4[i, ..., 0] + 1j * z4[i, ..., 1], O.zeta4_projected(d, edges, mmax)) < TOL


@pytest.mark.parametrize("odd", [False, True])
def test_full_row_tiles(ctx, odd):
    """Rows past one tile's 512, sets of l3 joined into one tile, rows no output takes."""
    n, nb, lmax = 16, 10, 4
    f = synth.lognormal_field(760, (n, n, n), 1.0, -2.0, dtype=np.float64)
    edges = np.linspace(0.5, 0.46 * n, nb + 1)
    d, _ = O.preprocess(f)
    z4 = ctx.full_odd(f, edges, lmax) if odd else ctx.full(f, edges, lmax4=lmax)[1]
    assert _err(z4, cpp.zeta4_full(d, edges, lmax, odd=odd)) < TOL
