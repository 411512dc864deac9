"""FP64 mechanics of strains so small that the squared residuals of a solve pass below 5.6e-309, where the
reciprocal of one is no longer finite (a quotient of two is): the model scales with the strain, so the
solve has to be that of ordinary strains times the scale.  The residuals' sums there hold some 40 bits."""
import numpy as np
import pytest

from paper_2203_16467_gb300.inputs import modulus_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", ["ISOTROPIC", "SPECTRAL", "VOLDEV"])
@pytest.mark.parametrize("power", [-300, -502])
def test_solution_scales_with_the_strain(split, power):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff
    n, out = 64, {}
    for k in (0, power):
        s = 2.0 ** k
        p = pff.Problem(n, n, pff.FP64, stream=torch.cuda.Stream().cuda_stream, E=modulus_field(n, n, 8.0, 1),
                        model=("AT1", split, "CRACK_SET"), params=dict(nu=0.2, ell=2.0))
        p.set_strain(None, (0.03 * s, 0.1 * s, 0.02 * s))
        rep = p.solve_mechanics()
        out[k] = (rep, p.get_fields(pff.FIELD_EPS_STAR) / s)
        p.close()
    (ra, a), (rb, b) = out[0], out[power]
    assert ra["status"] == rb["status"] == pff.OK
    assert abs(ra["mech_cg_iters"] - rb["mech_cg_iters"]) <= 1 and ra["newton_iters"] == rb["newton_iters"]
    assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(a)
