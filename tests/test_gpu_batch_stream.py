"""A batch step comes after what the caller has queued on the batch's stream, and before what it queues
next, also for the last group of a batch that had several (it keeps a stream of its own)."""
import numpy as np
import pytest

from paper_2203_16467_gb300.inputs import eps_M, gaussian_field, modulus_field

pytestmark = pytest.mark.gpu


class View:
    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr, "version": 2,
                                         "strides": None}


@pytest.mark.parametrize("n,mixed", [(64, True), (256, True), (64, False)])
def test_last_group_waits_for_the_batch_stream(n, mixed):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff
    prec, dtype = (pff.MIXED, torch.float32) if mixed else (pff.FP64, torch.float64)
    ell, em = 2.0, eps_M(1.0, 0.2, 1.0, 2.0)
    stream = torch.cuda.Stream()
    z = [gaussian_field(n, n, 3.0, k) for k in range(3)]
    phis = [torch.tensor(0.6 * ((x - x.min()) / (x.max() - x.min())) ** 2, dtype=dtype, device="cuda") for x in z]

    def make(st):
        p = pff.Problem(n, n, prec, stream=st.cuda_stream, E=modulus_field(n, n, 4.0, 1),
                        model=("AT1", "SPECTRAL", "CRACK_SET"), params=dict(nu=0.2, ell=ell))
        p.set_strain(None, (0.0, em, 0.0))
        ptr, f32 = p.get_device_ptr(pff.FIELD_PHI)
        return p, torch.as_tensor(View(ptr, (n, n), "<f4" if f32 else "<f8"), device="cuda")

    (p, phi), (other, _) = make(stream), make(stream)
    q, qphi = make(torch.cuda.Stream())
    b = pff.create_batch(2, 2 * pff.problem_bytes(n, n, prec), stream.cuda_stream)
    pff.batch_admit(b, p.h)
    slot = pff.batch_admit(b, other.h)
    pff.batch_set_group_size(b, 1)
    pff.batch_step(b, 2, 1)
    q.step_load(1)
    pff.batch_release(b, slot)
    pff.batch_step(b, 2, 1)          # one group from here on, its descriptor sent
    q.step_load(1)
    for k in range(3):
        with torch.cuda.stream(stream):
            torch.cuda._sleep(20_000_000)          # about ten milliseconds
            phi.copy_(phis[k])
        pff.batch_step(b, 2, 1)
        with torch.cuda.stream(stream):
            after = phi.clone()
        qphi.copy_(phis[k])
        torch.cuda.synchronize()
        q.step_load(1)
        np.testing.assert_array_equal(after.cpu().numpy(), qphi.cpu().numpy())
        np.testing.assert_array_equal(p.get_fields(pff.FIELD_EPS_STAR), q.get_fields(pff.FIELD_EPS_STAR))
    pff.destroy_batch(b)
    for x in (p, other, q):
        x.close()
