"""FP64 mechanics solves whose CG reads the tangent's frame stored by the Newton round: mean strains at the edges of
its encoding (coincident principal strains of either sign, one principal strain zero, opposite signs, both
negative, zero trace), in a medium that is uniform but for one inclusion, against the FP64 oracle.  Tolerance as for
the other solves at this mech_tol (tests/test_gpu_solvers.py)."""
import numpy as np
import pytest

from oracle import mechanics
from oracle.params import SPECTRAL, SPECTRAL_VOLDEV, VOLDEV, Params
from tests.helpers import bar3, tensor_rel_l2, to3

pytestmark = pytest.mark.gpu

MEANS = {"tension": (0.01, 0.01, 0.0), "compression": (-0.01, -0.01, 0.0), "uniaxial": (0.01, 0.0, 0.0),
         "uniaxial_compression": (0.0, -0.01, 0.0), "shear": (0.0, 0.0, 0.005), "opposite": (0.01, -0.002, 0.001),
         "both_negative": (-0.01, -0.003, 0.002)}


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    return m


@pytest.mark.parametrize("split", [SPECTRAL, VOLDEV, SPECTRAL_VOLDEV])
@pytest.mark.parametrize("mean", sorted(MEANS))
def test_mean_strains_at_the_edges(pff, split, mean):
    ny, nx = 32, 64
    E = np.ones((ny, nx))
    E[8:20, 10:30] = 2.0
    phi = np.zeros((ny, nx))
    phi[8:24, 20:40] = 0.4
    xx, yy, xy = MEANS[mean]
    eb = np.array([[xx, xy], [xy, yy]])
    par = Params(split=split, mech_tol=1e-10, mech_cg_rtol=1e-6)
    ref, _ = mechanics.solve(np.zeros((ny, nx, 2, 2)), eb, phi, E, par)
    p = pff.Problem(nx, ny, pff.FP64, E=E)
    p.set_model(par.fracture, par.split, par.irreversibility)
    p.set_params(nu=par.nu, Gc=par.Gc, ell=par.ell, dx=par.dx, mech_tol=par.mech_tol, mech_cg_rtol=par.mech_cg_rtol)
    p.set_phase_field(phi)
    p.set_strain(None, bar3(eb))
    rep = p.solve_mechanics()
    err = tensor_rel_l2(p.get_fields(pff.FIELD_STRAIN), to3(eb[None, None] + ref))
    assert err < 1e-8, (err, rep)
    p.close()
