"""The register-resident column passes (FP32 columns of 1024 and 2048 points) and the row passes of
256 points on, through the operator entry points against the FP64 oracle: mode columns that do not
fill the last block (nx = 16, 64), one row block to many, both component counts.  Tolerances as for
the other sizes of the operators (tests/test_gpu_ops.py)."""
import numpy as np
import pytest

from oracle import fourier
from paper_2203_16467_gb300.inputs import gaussian_field
from tests.helpers import from3, rel_l2, tensor_rel_l2, to3

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    return m


def _field(ny, nx, seed):
    return gaussian_field(ny, nx, max(2.0, nx / 16), seed) + 0.3 * np.random.default_rng(seed).standard_normal((ny, nx))


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("ny,nx", [(1024, 16), (1024, 64), (2048, 16), (2048, 64), (1024, 256), (16, 1024), (16, 2048),
                                   (1024, 1024)])
def test_operators(pff, prec, ny, nx):
    tol = 1e-12 if prec == 0 else (3e-6 if nx * ny <= 256 * 256 else 1e-5)
    p = pff.Problem(nx, ny, prec)
    g = _field(ny, nx, 1)
    assert rel_l2(p.apply_laplacian(g), fourier.laplacian(g)) < tol
    z = np.stack([_field(ny, nx, s) for s in (2, 3, 4)])
    assert tensor_rel_l2(p.apply_projection(z), to3(fourier.project(from3(z)))) < tol
    p.close()
