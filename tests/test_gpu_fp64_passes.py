"""The FP64 passes at the edges of their block shapes: one column per block from 256 points on (the last block's
column is the Nyquist mode), two below (a last block that is half padding), rows of 256 values per block up to 256
points, and the tangential form of the projection (idempotent, exact on the axes' modes up to rounding).

Tolerance: two 2-D FFTs of log2(N) <= 22 stages at a unit roundoff of 1.1e-16, one to two roundoffs a stage, and the
multiplier's ten: below 1e-14 of the norm; taken with a margin of ten."""
import numpy as np
import pytest

from oracle import fourier
from tests.helpers import from3, rel_l2, tensor_rel_l2, to3

pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    return m


@pytest.mark.parametrize("ny,nx", [(16, 16), (128, 16), (256, 16), (512, 16), (128, 256), (256, 128), (256, 256),
                                   (16, 512), (512, 512), (2048, 16), (1024, 2048)])
def test_operators(pff, ny, nx):
    rng = np.random.default_rng(ny + 3 * nx)
    p = pff.Problem(nx, ny, pff.FP64)
    g = rng.standard_normal((ny, nx))
    assert rel_l2(p.apply_laplacian(g), fourier.laplacian(g)) < TOL
    z = rng.standard_normal((3, ny, nx))
    z[0] += 5.0 * np.cos(2 * np.pi * np.arange(nx) / nx)[None, :]      # modes on either axis
    z[1] += 5.0 * np.cos(2 * np.pi * np.arange(ny) / ny)[:, None]
    out = p.apply_projection(z)
    assert tensor_rel_l2(out, to3(fourier.project(from3(z)))) < TOL
    assert tensor_rel_l2(p.apply_projection(out), out) < TOL
    p.close()
