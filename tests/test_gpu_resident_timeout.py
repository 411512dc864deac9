"""The one-launch solves of small FP32 grids (and the persistent one of 512^2 in steps and batches) when a
wait between their blocks runs out: a limit of one
cycle ends the first wait for which the bytes are not there yet.  The calls report
PFF_ERR_BARRIER_TIMEOUT, apply nothing of the given-up solve, and the handle then solves as a fresh
one does.  The sizes have CTAs with and without mode columns, one and several rows per warp."""
import ctypes

import numpy as np
import pytest

from paper_2203_16467_gb300.inputs import eps_M, gaussian_field, modulus_field

pytestmark = pytest.mark.gpu

SIZES = [(16, 16), (64, 64), (128, 128), (256, 32)]
ELL = 2.0


@pytest.fixture(scope="module")
def pff():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff as m
    yield m
    m.set_barrier_spin_limit(0)


def make(pff, nx, ny, load=1.1, seed=1, **kw):
    import torch
    em = eps_M(1.0, 0.2, 1.0, ELL)
    z = gaussian_field(ny, nx, 3.0, 2)
    p = pff.Problem(nx, ny, pff.MIXED, stream=torch.cuda.Stream().cuda_stream, E=modulus_field(ny, nx, 4.0, seed),
                    model=("AT1", "SPECTRAL", "CRACK_SET"), params=dict(nu=0.2, ell=ELL, d_eps_bar=(0.0, em / 20, 0.0), **kw))
    p.set_phase_field(0.8 * ((z - z.min()) / (z.max() - z.min())) ** 2)
    p.set_strain(None, (0.1 * em, load * em, 0.05 * em))
    return p


def state(pff, p):
    return p.get_fields(pff.FIELD_PHI), p.get_fields(pff.FIELD_EPS_STAR)


def same(a, b):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("call", ["pff_solve_mechanics", "pff_solve_phase_field"])
def test_sub_problem(pff, nx, ny, call):
    p, q = make(pff, nx, ny), make(pff, nx, ny)
    before = state(pff, p)
    pff.set_barrier_spin_limit(1)
    rc = getattr(pff.lib, call)(p.h, ctypes.byref(pff.StepReport()))
    pff.set_barrier_spin_limit(0)
    assert rc == pff.ERR_BARRIER_TIMEOUT
    assert "timed out" in pff.lib.pff_last_error(p.h).decode()
    same(state(pff, p), before)
    for x in (p, q):
        assert getattr(pff.lib, call)(x.h, ctypes.byref(pff.StepReport())) == pff.OK
    same(state(pff, p), state(pff, q))
    p.close()
    q.close()


@pytest.mark.parametrize("evolution", [0, 1, 2])
def test_load_step(pff, evolution):
    p, q = make(pff, 64, 64, evolution=evolution), make(pff, 64, 64, evolution=evolution)
    before = state(pff, p)
    reps, done = (pff.StepReport * 2)(), ctypes.c_int(7)
    pff.set_barrier_spin_limit(1)
    rc = pff.lib.pff_step_load(p.h, 2, reps, ctypes.byref(done))
    pff.set_barrier_spin_limit(0)
    assert rc == pff.ERR_BARRIER_TIMEOUT and done.value == 0
    same(state(pff, p), before)
    em = eps_M(1.0, 0.2, 1.0, ELL)
    for x in (p, q):   # (an alternating-minimisation increment has been added)
        x.set_strain(None, (0.1 * em, 1.1 * em, 0.05 * em))
        x.step_load(1)
    same(state(pff, p), state(pff, q))
    p.close()
    q.close()


def test_batch(pff):
    import torch
    n = 64
    stream = torch.cuda.Stream()
    probs = [make(pff, n, n, 1.05 + 0.1 * k, k) for k in range(2)]
    b = pff.create_batch(2, 2 * pff.problem_bytes(n, n, pff.MIXED), stream.cuda_stream)
    for p in probs:
        pff.batch_admit(b, p.h)
    before = [state(pff, p) for p in probs]
    reps, done = (pff.StepReport * 6)(), (ctypes.c_int * 2)(7, 7)
    pff.set_barrier_spin_limit(1)
    rc = pff.lib.pff_batch_step(b, 3, reps, done)
    pff.set_barrier_spin_limit(0)
    assert rc == pff.ERR_BARRIER_TIMEOUT and list(done) == [0, 0]
    assert reps[0].status == reps[3].status == pff.ERR_BARRIER_TIMEOUT
    for p, s in zip(probs, before):
        same(state(pff, p), s)
    pff.batch_step(b, 2, 1)
    for k, p in enumerate(probs):
        q = make(pff, n, n, 1.05 + 0.1 * k, k)
        q.step_load(1)
        same(state(pff, p), state(pff, q))
        q.close()
    pff.destroy_batch(b)
    for p in probs:
        p.close()


@pytest.mark.parametrize("nx,ny", SIZES)
def test_laplacian_leaves_nan(pff, nx, ny):
    import torch
    x = torch.randn(ny, nx, device="cuda")
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def lap(out):
        assert pff.lib.pff_apply_laplacian_noalloc_f32(nx, ny, 1.0, ctypes.c_void_p(x.data_ptr()),
                                                       ctypes.c_void_p(out.data_ptr()), st, None) == 0
        torch.cuda.synchronize()

    pff.set_barrier_spin_limit(1)
    lap(y)
    pff.set_barrier_spin_limit(0)
    lap(z)
    assert torch.isnan(y).all()
    assert torch.isfinite(z).all() and z.abs().max() > 0


def test_persistent_step_and_batch(pff):
    import torch
    n = 512
    try:
        pff.set_persistent(True)
        p = make(pff, n, n)
        before = p.get_fields(pff.FIELD_PHI)
        done = ctypes.c_int(7)
        pff.set_barrier_spin_limit(1)
        rc = pff.lib.pff_step_load(p.h, 2, (pff.StepReport * 2)(), ctypes.byref(done))
        pff.set_barrier_spin_limit(0)
        assert rc == pff.ERR_BARRIER_TIMEOUT and done.value == 0
        np.testing.assert_array_equal(p.get_fields(pff.FIELD_PHI), before)
        assert len(p.step_load(1)) == 1
        # a batch with a small grid of FP64 beside it, whose solves have no such waits: its step counts
        small = pff.Problem(32, 32, pff.FP64, params=dict(nu=0.2, ell=ELL))
        small.set_strain(None, (0.0, 1.0, 0.0))
        b = pff.create_batch(2, pff.problem_bytes(n, n, pff.MIXED) + pff.problem_bytes(32, 32, pff.FP64),
                             torch.cuda.Stream().cuda_stream)
        for x in (p, small):
            pff.batch_admit(b, x.h)
        before = p.get_fields(pff.FIELD_PHI)
        reps, done = (pff.StepReport * 4)(), (ctypes.c_int * 2)(7, 7)
        pff.set_barrier_spin_limit(1)
        rc = pff.lib.pff_batch_step(b, 2, reps, done)
        pff.set_barrier_spin_limit(0)
        assert rc == pff.ERR_BARRIER_TIMEOUT and list(done) == [0, 1]
        assert reps[0].status == pff.ERR_BARRIER_TIMEOUT and reps[2].status == pff.OK and reps[2].bccg_iters > 0
        np.testing.assert_array_equal(p.get_fields(pff.FIELD_PHI), before)
        pff.destroy_batch(b)
        p.close()
        small.close()
    finally:
        pff.set_barrier_spin_limit(0)
        pff.set_persistent(False)
