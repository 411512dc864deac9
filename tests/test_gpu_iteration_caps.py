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


def both_paths(pff, run):
    """The one-launch solve and, with kernel timing on, the per-kernel path on the same problem."""
    out = []
    try:
        for per_kernel in (False, True):
            pff.timing_enable(per_kernel)
            out.append(run())
    finally:
        pff.timing_enable(False)
    return out


def close(a, b):   # either path is held to 1e-5 of the oracle
    assert np.linalg.norm(a - b) <= 2e-5 * np.linalg.norm(b)


@pytest.mark.parametrize("n", [16, 64, 128])
@pytest.mark.parametrize("caps", [dict(mech_max_cg=4, mech_max_newton=3), dict(mech_max_newton=1),
                                  dict(mech_max_cg=1, mech_max_newton=2)])
def test_mechanics_caps(pff, n, caps):
    def run():
        p = make(pff, n, 1, **caps)
        r = p.solve_mechanics()
        e = p.get_fields(pff.FIELD_STRAIN)
        p.close()
        return r, e
    (ra, ea), (rb, eb) = both_paths(pff, run)
    assert ra["status"] == rb["status"] == pff.ERR_NOT_CONVERGED
    assert ra["newton_iters"] == rb["newton_iters"] == caps["mech_max_newton"]
    if "mech_max_cg" in caps:
        assert ra["mech_cg_iters"] == rb["mech_cg_iters"] == caps["mech_max_cg"] * caps["mech_max_newton"]
    close(ea, eb)


@pytest.mark.parametrize("n", [16, 64, 128])
@pytest.mark.parametrize("cap", [1, 2, 9])
def test_phase_field_caps(pff, n, cap):
    def run():
        p = make(pff, n, 1, pf_max_iter=cap)
        r = p.solve_phase_field()
        phi = p.get_fields(pff.FIELD_PHI)
        p.close()
        return r, phi
    (ra, pa), (rb, pb) = both_paths(pff, run)
    assert ra["status"] == rb["status"] == pff.ERR_NOT_CONVERGED
    assert ra["bccg_iters"] == rb["bccg_iters"] == cap
    # a value at its bound may be clamped in one path and just not in the other
    assert abs(ra["bccg_clamp_iters"] - rb["bccg_clamp_iters"]) <= 2
    assert abs(ra["bccg_full_iters"] - rb["bccg_full_iters"]) <= 2
    assert abs(ra["n_active"] - rb["n_active"]) <= n * n // 100
    close(pa, pb)


def long_solve(pff, n, tol):
    """An AT2 solve from the undamaged state, of which an early overshoot at most is clamped."""
    import torch
    em = eps_M(1.0, 0.2, 1.0, 2.0)
    z = gaussian_field(n, n, 2.0, 3)
    p = pff.Problem(n, n, 1, stream=torch.cuda.Stream().cuda_stream, E=modulus_field(n, n, 2.0, 1),
                    model=("AT2", "ISOTROPIC", "DAMAGE"), params=dict(nu=0.2, ell=4.0, pf_tol=tol, pf_atol=0.0))
    p.set_strain(em * np.stack([8.0 * z, 4.0 * np.roll(z, 3, 0), 0.0 * z]), (0.0, em, 0.0))
    r = p.solve_phase_field()
    phi = p.get_fields(pff.FIELD_PHI)
    p.close()
    return r, phi


@pytest.mark.parametrize("n", [32, 64, 128])
def test_refresh_and_confirmation(pff, n):
    # an explicit residual where a value was clamped, after 31 iterations without one, and to confirm the end
    (ra, _), (rb, _) = both_paths(pff, lambda: long_solve(pff, n, 1e-4))
    for r in (ra, rb):
        its, full, clamped = r["bccg_iters"], r["bccg_full_iters"], r["bccg_clamp_iters"]
        assert r["status"] == pff.OK and clamped <= 2
        assert max(clamped, 1 + its // 33) <= full <= clamped + 2 + its // 32
    assert abs(ra["bccg_iters"] - rb["bccg_iters"]) <= 2


@pytest.mark.parametrize("n", [32, 64, 128])
def test_stall(pff, n):
    # a tolerance below the rounding level of the residual: the solve ends by itself and has converged to that level
    (ra, pa), (rb, pb) = both_paths(pff, lambda: long_solve(pff, n, 1e-30))
    assert ra["status"] == rb["status"] == pff.OK
    assert min(ra["bccg_iters"], rb["bccg_iters"]) > 64
    close(pa, pb)
