"""The driving-force maximum of a load step (Algorithm 4 lines 4-10) screens pixels in FP32 and
evaluates only candidates in FP64: its results must be the FP64 maxima over all pixels, the first
maximiser on ties, at the smallest grid, one and several pixels per thread, and for values near
the ends of the FP32 range (strains of 1e-20, moduli of 1e20), where nothing is screened out."""
import numpy as np
import pytest

from oracle import constitutive as cm
from oracle.fourier import laplacian
from oracle.params import ISOTROPIC, SPECTRAL, VOLDEV
from paper_2203_16467_gb300.inputs import gaussian_field, modulus_field
from tests.helpers import from3

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    return m


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("split,name", [(SPECTRAL, "SPECTRAL"), (ISOTROPIC, "ISOTROPIC"), (VOLDEV, "VOLDEV")])
@pytest.mark.parametrize("ny,nx,strain,E0", [(16, 16, 1e-2, 1.0), (256, 256, 1e-2, 1.0), (512, 256, 1e-2, 1.0),
                                             (32, 64, 1e-20, 1.0), (32, 64, 1e-2, 1e20)])
def test_maxima_are_the_fp64_maxima(pff, prec, split, name, ny, nx, strain, E0):
    E = E0 * modulus_field(ny, nx, 4.0, 1)
    z = gaussian_field(ny, nx, 4.0, 2)
    phi = 0.5 * (z - z.min()) / (z.max() - z.min())
    if prec == 1:
        E, phi = E.astype(np.float32).astype(float), phi.astype(np.float32).astype(float)
    p = pff.Problem(nx, ny, prec, E=E, model=("AT1", name, "CRACK_SET"),
                    params=dict(nu=0.2, Gc=1.0, ell=2.0, F_max=1e300, mech_tol=1e-4, pf_max_iter=1))
    p.set_phase_field(phi)
    p.set_strain(None, (0.2 * strain, strain, 0.1 * strain))
    rep = p.step_load(1)[0]
    assert rep["gamma"] == 1.0
    eps = np.array(rep["eps_bar"])[:, None, None] + p.get_fields(pff.FIELD_EPS_STAR)
    lam, mu = cm.lame(E, 0.2)
    psi = cm.psi_plus(from3(eps), lam, mu, split)
    c = 1.0 / (8.0 / 3.0 * 2.0)
    D = 2.0 * (1.0 - phi) * psi
    v = D - c + 2.0 * c * 4.0 * laplacian(phi)
    # FP64 problems: to rounding; mixed ones: nabla^2 phi is an FP32 field (relative 1e-5 of its largest value)
    tol = 1e-11 * np.abs(v).max() if prec == 0 else 1e-5 * (2.0 * c * 4.0 * np.abs(laplacian(phi)).max()) + 1e-11 * np.abs(v).max()
    assert abs(rep["mF_max"] - v.max()) <= tol
    assert v.ravel()[rep["istar"]] >= v.max() - 2 * tol
    np.testing.assert_allclose(rep["D_max"], D.max(), rtol=1e-11, atol=0)
    p.close()


@pytest.mark.parametrize("n", [16, 256, 512])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_first_maximiser_on_ties(pff, prec, n):
    # a homogeneous undamaged grid: every pixel holds the maximum
    p = pff.Problem(n, n, prec, model=("AT1", "SPECTRAL", "CRACK_SET"), params=dict(nu=0.2, ell=2.0))
    p.set_strain(None, (0.0, 0.1, 0.0))
    rep = p.step_load(1)[0]
    assert rep["istar"] == 0
    p.close()
