"""Which calls take the integer-product transforms, and what the others need not pay."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from test_gpu_digit_transform import TOL, _problem  # noqa: E402

pytestmark = pytest.mark.gpu


def test_capture_before_the_first_transform():
    """A capture of FP64 single steps whose staging exists already, but not the
    digits' buffers: nothing may be allocated there."""
    op, _, f, dev = _problem(64, 256, 1, 0)
    x = torch.randn((1, 64, 256), dtype=torch.float64, device=dev)
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    try:
        P.ax_apply_operator(op, x, y, 1)  # makes the staging
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            P.ax_apply_dst(op, x, y, 64)
            P.ax_apply_dst_inverse(op, y, z, 64)
        g.replay()
        torch.cuda.synchronize()
        assert (z - x).norm() <= 2 * TOL * x.norm()
        P.ax_apply_dst(op, x, z, 64)  # outside a capture: the digits
        assert (z - y).norm() <= 2 * TOL * x.norm()
        g.replay()
        torch.cuda.synchronize()
        P.ax_apply_preconditioner(op, x, y, 1)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            P.ax_apply_preconditioner(op, x, z, 1)
        # a larger solve on the operator leaves the captured staging alone
        fm = torch.from_numpy(np.repeat(f[:1], 4, 0)).to(dev)
        P.ax_solve(op, fm, torch.zeros_like(fm), 4, 1e-8, 500, P.AX_PCG_FP64)
        z.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, z)
    finally:
        P.ax_destroy_operator(op)


def test_many_right_hand_sides():
    """More right-hand sides than a grid dimension y holds blocks."""
    m, nr, nz = 65536, 48, 128
    op, _, _, dev = _problem(nr, nz, 1, 0)
    x = torch.randn((nr, nz), dtype=torch.float64, device=dev).expand(m, nr, nz).contiguous()
    x[m - 1] *= 2.0
    y = torch.zeros_like(x)
    try:
        P.ax_apply_preconditioner(op, x, y, m)
        assert torch.equal(y[1], y[0]) and torch.equal(y[m - 2], y[0]) and torch.equal(y[m - 1], 2.0 * y[0])
        one = torch.zeros_like(x[:1])
        P.ax_apply_preconditioner(op, x[:1], one, 1)
        assert (one[0] - y[0]).norm() <= 1e-12 * one.norm()
    finally:
        P.ax_destroy_operator(op)
        del x, y
        torch.cuda.empty_cache()


def test_chebyshev_solves_hold_no_digits():
    """AX_CHEB_FP64 transforms by FFT: the digits' 16 bytes per point are first
    allocated by the AX_PCG_FP64 solve after it, whose vectors exist by then."""
    nr, nz, m = 256, 511, 32
    op, _, f, dev = _problem(nr, nz, 1, 0)
    fd = torch.from_numpy(np.repeat(f[:1], m, 0)).to(dev)
    u = torch.zeros_like(fd)
    free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]  # noqa: E731
    try:
        st, _ = P.ax_solve(op, fd, u, m, 1e-6, 500, P.AX_CHEB_FP64)
        assert st == P.AX_OK
        before = free()
        st, _ = P.ax_solve(op, fd, u, m, 1e-6, 500, P.AX_PCG_FP64)
        assert st == P.AX_OK
        assert before - free() >= 16 * nr * nz * m
    finally:
        P.ax_destroy_operator(op)
