"""pff_apply_laplacian_noalloc_f32 over the sizes that take one cluster launch (up to 2^14 pixels) and the first
beyond: against the FP64 entry point, against the three-pass path (which a field off the 8-byte boundary takes),
in place, and replayed from a captured graph."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDES = (16, 32, 64, 128, 256)
SMALL = [(ny, nx) for ny in SIDES for nx in SIDES if nx * ny <= 1 << 14] + [(128, 256), (256, 128), (16, 512), (512, 16)]


@pytest.fixture(scope="module")
def env():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    from paper_2203_16467_gb300 import pff
    assert torch.cuda.is_available()
    return pff, torch


def _lap(pff, torch, src, dst, nx, ny, dx, name="pff_apply_laplacian_noalloc_f32"):
    msg = ctypes.c_char_p()
    rc = getattr(pff.lib, name)(nx, ny, dx, ctypes.c_void_p(src.data_ptr()), ctypes.c_void_p(dst.data_ptr()),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), ctypes.byref(msg))
    assert rc == pff.OK, msg.value


# Tolerance: two FFTs of log2(N) <= 14 stages each at a unit roundoff of 6e-8 add about sqrt(2 * 14) roundoffs
# per mode of white noise, whose norm the highest modes carry: 3e-7, taken six times.
TOL = 2e-6


@pytest.mark.parametrize("ny,nx", SMALL)
def test_small_fields(env, ny, nx):
    pff, torch = env
    dx = 0.5
    rng = np.random.default_rng(7 * nx + ny)
    with torch.cuda.stream(torch.cuda.Stream()):
        src64 = torch.tensor(rng.standard_normal((ny, nx)), dtype=torch.float64, device="cuda")
        ref = torch.empty_like(src64)
        _lap(pff, torch, src64.float().double(), ref, nx, ny, dx, "pff_apply_laplacian_noalloc")
        src = src64.float()
        out = torch.full_like(src, float("nan"))
        n0 = pff.kernel_launches()
        _lap(pff, torch, src, out, nx, ny, dx)
        small = nx * ny <= 1 << 14 and max(nx, ny) <= 256
        assert pff.kernel_launches() - n0 == (1 if small else 3)

        # one float off the boundary: scalar accesses, three passes
        buf = torch.zeros(nx * ny + 2, device="cuda")
        buf2 = torch.full((nx * ny + 2,), float("nan"), device="cuda")
        off, off_out = buf[1:-1], buf2[1:-1]
        off.copy_(src.flatten())
        n0 = pff.kernel_launches()
        _lap(pff, torch, off, off_out, nx, ny, dx)
        assert pff.kernel_launches() - n0 == 3
        assert bool(torch.isnan(buf2[0])) and bool(torch.isnan(buf2[-1]))

        place = src.clone()
        _lap(pff, torch, place, place, nx, ny, dx)

        # a captured call computes from the input's contents at each replay
        gin, gout = torch.zeros_like(src), torch.full_like(src, float("nan"))
        torch.cuda.current_stream().synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _lap(pff, torch, gin, gout, nx, ny, dx)
        gin.copy_(src)
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        n = ref.norm()
        for got in (out.double(), off_out.double().view(ny, nx), place.double(), gout.double()):
            assert float((got - ref).norm() / n) < TOL
        assert torch.equal(out, place) and torch.equal(out, gout)


def test_non_finite_values_spread_as_in_the_three_passes(env):
    pff, torch = env
    with torch.cuda.stream(torch.cuda.Stream()):
        src = torch.zeros(64, 64, device="cuda")
        src[3, 5] = float("nan")
        out = torch.zeros_like(src)
        _lap(pff, torch, src, out, 64, 64, 1.0)
        assert bool(torch.isnan(out).all())
