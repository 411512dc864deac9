"""The iteration caps of the sub-problem solves: any positive int is a cap (a huge one stands for none),
and a solve that reaches its cap says so, in the one-launch solves, the per-kernel path and FP64 alike."""
import numpy as np
import pytest

from paper_2203_16467_gb300.inputs import eps_M, gaussian_field, modulus_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    return m


def make(pff, n, prec, **kw):
    import torch
    em = eps_M(1.0, 0.2, 1.0, 2.0)
    z = gaussian_field(n, n, 3.0, 2)
    p = pff.Problem(n, n, prec, stream=torch.cuda.Stream().cuda_stream, E=modulus_field(n, n, 4.0, 1),
                    model=("AT1", "SPECTRAL", "CRACK_SET"), params=dict(nu=0.2, ell=2.0, **kw))
    p.set_phase_field(0.8 * ((z - z.min()) / (z.max() - z.min())) ** 2)
    p.set_strain(None, (0.1 * em, 1.1 * em, 0.05 * em))
    return p


@pytest.mark.parametrize("cap", [2**30 - 1, 2**30, 2**30 + 1, 2**31 - 1])
@pytest.mark.parametrize("n,prec", [(64, 1), (256, 1), (64, 0)])
def test_a_huge_cap_is_no_cap(pff, n, prec, cap):
    p, q = make(pff, n, prec, pf_max_iter=cap), make(pff, n, prec)
    rp, rq = p.solve_phase_field(), q.solve_phase_field()
    assert rq["bccg_iters"] > 0 and rp["bccg_iters"] == rq["bccg_iters"] and rp["status"] == pff.OK
    np.testing.assert_array_equal(p.get_fields(pff.FIELD_PHI), q.get_fields(pff.FIELD_PHI))
    p.close()
    q.close()
