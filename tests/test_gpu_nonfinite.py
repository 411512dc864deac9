"""A mechanics solve whose residual is not a number has not converged, whichever path runs it: the
per-kernel path of either precision, the one-launch solve of small grids, the cluster solve of 512^2."""
import ctypes

import pytest

from paper_2203_16467_gb300.inputs import eps_M, modulus_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("path", ["resident", "kernels", "fp64", "cluster"])
@pytest.mark.parametrize("split", ["SPECTRAL", "VOLDEV"])
@pytest.mark.parametrize("where", ["eps_bar", "eps_star"])
def test_nan_is_not_converged(path, split, where):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2203_16467_gb300 import pff
    n = 512 if path == "cluster" else 64
    em = eps_M(1.0, 0.2, 1.0, 2.0)
    nan = float("nan")
    star = torch.zeros(3, n, n, dtype=torch.float64, device="cuda")
    if where == "eps_star":
        star[1, 3, 5] = nan
    try:
        pff.timing_enable(path == "kernels")
        pff.set_cluster_mechanics(path == "cluster")
        p = pff.Problem(n, n, pff.FP64 if path == "fp64" else pff.MIXED, stream=torch.cuda.Stream().cuda_stream,
                        E=modulus_field(n, n, 8.0, 1), model=("AT1", split, "CRACK_SET"),
                        params=dict(nu=0.2, ell=2.0, mech_max_newton=3))
        p.set_strain(star, (0.0, nan if where == "eps_bar" else em, 0.0))
        rep = pff.StepReport()
        assert pff.lib.pff_solve_mechanics(p.h, ctypes.byref(rep)) == pff.ERR_NOT_CONVERGED
        assert rep.status == pff.ERR_NOT_CONVERGED
        p.close()
    finally:
        pff.timing_enable(False)
        pff.set_cluster_mechanics(False)
