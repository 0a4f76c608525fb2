"""Thousands of right-hand sides on a small grid: workspace and results.

256 KB of partial sums per right-hand side and, on 15 x 15 (transforms by FFT), at most 38
KB of vectors: at most 320 KB.  A larger grid, whose kernels' sums need whole rows,
checks that they do not run into each other.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from test_gpu_digit_transform import _problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [P.AX_PCG_FP64, P.AX_PCG_MIXED, P.AX_CHEB_MIXED])
def test_many_right_hand_sides_of_a_small_grid(method):
    m, n = 4096, 15
    op, ora, f, dev = _problem(n, n, 8, 0)
    fd = torch.from_numpy(np.resize(f, (m, n, n))).to(dev)
    u = torch.zeros_like(fd)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    try:
        st, _ = P.ax_solve(op, fd, u, m, 1e-10, 500, method)
        assert st == P.AX_OK
        assert before - torch.cuda.mem_get_info()[0] <= m * 320 * 1024
        un = u.cpu().numpy()
        assert np.array_equal(un[8:], un[:-8])
        for j in range(8):
            phi = ora.phi(f[j])
            assert np.linalg.norm(phi - ora.apply_A(un[j])) <= 1.01e-10 * np.linalg.norm(phi)
    finally:
        P.ax_destroy_operator(op)


@pytest.mark.parametrize("nr,nz", [(3000, 3000), (4200, 4300)])
def test_grids_on_both_sides_of_half_a_row(nr, nz):
    """(4512 and 8942 stencil sums.)"""
    op, ora, f, dev = _problem(nr, nz, 1, 0)
    fd = torch.from_numpy(f[:1]).to(dev)
    u = torch.zeros_like(fd)
    try:
        st, _ = P.ax_solve(op, fd, u, 1, 1e-8, 500, P.AX_PCG_MIXED)
        assert st == P.AX_OK
        phi = ora.phi(f[0])
        assert np.linalg.norm(phi - ora.apply_A(u[0].cpu().numpy())) <= 1.01e-8 * np.linalg.norm(phi)
    finally:
        P.ax_destroy_operator(op)
