"""The BCCG start of FP32 problems: its diagonal a = eta/dt + 2 psi_0^+ + c f'' and right-hand side
b = 2 (1 - phi) psi_0^+ - c f' + kappa nabla^2 phi are the FP64 values (those of an FP64 problem with the
same inputs, which the oracle confirms) rounded once, also where b is a small difference of its terms.
Both planes stay in the problem after a phase-field solve (the planes of a problem lie at equal
distances: 7 and 8 after phi).  phi is uniform, so that nabla^2 phi, an FP32 transform, is 0."""
import numpy as np
import pytest

from oracle import constitutive as cm
from oracle.params import ISOTROPIC, SPECTRAL, VOLDEV
from paper_2203_16467_gb300.inputs import gaussian_field
from tests.helpers import from3

pytestmark = pytest.mark.gpu
NU, ELL = 0.2, 2.0


class View:
    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (n, n), "typestr": typestr, "version": 2,
                                         "strides": None}


@pytest.mark.parametrize("split,name", [(SPECTRAL, "SPECTRAL"), (ISOTROPIC, "ISOTROPIC"), (VOLDEV, "VOLDEV")])
@pytest.mark.parametrize("fracture", ["AT1", "AT2"])
@pytest.mark.parametrize("near", [0.0, 1e-3, 1e-6])     # size of b against its terms (0: as large)
@pytest.mark.parametrize("strain", [0.4, 1e-9])
def test_a_and_b_are_fp64_values(split, name, fracture, near, strain):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff
    n, phi0 = 256, float(np.float32(0.3))
    f32 = lambda x: np.asarray(x, dtype=np.float32).astype(np.float64)  # noqa: E731
    z = gaussian_field(n, n, 4.0, 3)
    bar = np.array([0.3 * strain, strain, 0.1 * strain])
    es = f32(strain * np.stack([0.2 * z, 0.1 * np.roll(z, 5, 0), 0.1 * np.roll(z, 9, 1)]))
    eps = from3(bar[:, None, None] + es)
    c = 1.0 / ((8.0 / 3.0 if fracture == "AT1" else 2.0) * ELL)
    cf = c * (1.0 if fracture == "AT1" else 2.0 * phi0)
    unit = cm.psi_plus(eps, *cm.lame(np.ones((n, n)), NU), split)   # psi_0^+ of E = 1
    E = f32(cf / (2.0 * (1.0 - phi0) * unit) * (1.0 + near * z) if near else 1.0 + 0.2 * np.abs(z))
    lam, mu = cm.lame(E, NU)
    psi = cm.psi_plus(eps, lam, mu, split)
    want = 2.0 ** -16 / ELL + 2.0 * psi + (0.0 if fracture == "AT1" else 2.0 * c), 2.0 * (1.0 - phi0) * psi - cf
    got = {}
    for prec, kind in ((pff.MIXED, "<f4"), (pff.FP64, "<f8")):
        p = pff.Problem(n, n, prec, E=E, model=(fracture, name, "DAMAGE"), params=dict(nu=NU, ell=ELL, pf_max_iter=1))
        p.set_phase_field(np.full((n, n), phi0))
        p.set_strain(es, bar)
        p.solve_phase_field()
        torch.cuda.synchronize()
        ptr, nxt = (p.get_device_ptr(w)[0] for w in (pff.FIELD_PHI, pff.FIELD_EPS_STAR))
        got[prec] = [torch.as_tensor(View(ptr + k * (nxt - ptr), n, kind), device="cuda").cpu().numpy() for k in (7, 8)]
        p.close()
    M2 = np.max(np.abs(bar)[:, None, None] + np.abs(es), axis=0) ** 2
    terms = 2.0 * (2.0 * lam + 10.0 * mu) * M2 + cf
    for x, v, w in zip(got[pff.MIXED], got[pff.FP64], want):
        assert np.all(np.abs(v - w) <= 32 * 2.0 ** -53 * terms)     # some 13 roundings on each side
        # the same FP64 formula, compiled twice: products may be contracted otherwise, a rounding's difference
        d = 2.0 ** -53 * terms
        lo, hi = (v - d).astype(np.float32), (v + d).astype(np.float32)
        assert np.all((lo <= x) & (x <= hi)), int(np.sum((x < lo) | (x > hi)))
