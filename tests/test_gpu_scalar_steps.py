"""Scalar steps taken by a kernel's last CTA, and the strip kernels' edges.

  - one operator solved to a loose, then to a tight tolerance (and the reverse)
    meets each in the oracle's FP64 true residual: the captured iterations
    read the tolerance of the current solve;
  - mixed solves on grids whose rows and columns end inside a strip (2 rows x 128
    columns per warp, 4 or 8 warps per CTA) or a 8 x 32 update patch meet the
    tolerance, and a right-hand side solved alone gives the bits it gives among
    nine (groups of 8 share a CTA's coefficients).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_1002_3094_gb300 as P  # noqa: E402
from paper_1002_3094_gb300.inputs import sample_operator_inputs, sample_rhs  # noqa: E402
from workloads import layered_inclusion_medium  # noqa: E402

pytestmark = pytest.mark.gpu


def _problem(nr, nz, m, bc_z=0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    med = layered_inclusion_medium(n_rhs=m, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz, bc_z=bc_z)
    dev = torch.device("cuda:0")
    op = P.ax_setup_operator(*[torch.from_numpy(x).to(dev) for x in (kr, kz, q)], nr, nz, bc_z=bc_z)
    return op, O.Operator(kr, kz, q, O.Grid(nr, nz, bc_z=bc_z)), sample_rhs(med, nr, nz, bc_z=bc_z), dev


def _rel(ora, f, u):
    phi = ora.phi(f)
    return np.linalg.norm(phi - ora.apply_A(u)) / np.linalg.norm(phi)


@pytest.mark.parametrize("method", [P.AX_PCG_MIXED, P.AX_PCG_FP64])
@pytest.mark.parametrize("tols", [(1e-3, 1e-10), (1e-10, 1e-3, 1e-9)])
def test_each_solve_meets_its_own_tolerance(method, tols):
    op, ora, f, dev = _problem(96, 72, 2)
    fd = torch.from_numpy(f).to(dev)
    try:
        for _ in range(3):  # launched directly first, then as a captured graph
            for tol in tols:
                u = torch.zeros_like(fd)
                st, _ = P.ax_solve(op, fd, u, 2, tol, 2000, method)
                assert st == P.AX_OK
                for j in range(2):
                    assert _rel(ora, f[j], u[j].cpu().numpy()) <= tol, (tol, j)
    finally:
        P.ax_destroy_operator(op)


# the last two have one right-hand side below and nine above the tile count at
# which the tensor-core transform takes its 32-column tiles
@pytest.mark.parametrize("bc_z", [0, 1])
@pytest.mark.parametrize("nr,nz", [(1, 5), (2, 128), (3, 129), (17, 131), (40, 256), (64, 33), (65, 260), (259, 127),
                                   (513, 517), (900, 386)])
def test_strip_edges(nr, nz, bc_z):
    m = 9
    op, ora, f, dev = _problem(nr, nz, m, bc_z)
    fd = torch.from_numpy(f).to(dev)
    try:
        for tc in (0, 1):
            P.ax_set_option(op, "dst_tensor", tc)
            u = torch.zeros_like(fd)
            st, _ = P.ax_solve(op, fd, u, m, 1e-8, 2000, P.AX_PCG_MIXED)
            assert st == P.AX_OK
            un = u.cpu().numpy()
            for j in range(m):
                assert _rel(ora, f[j], un[j]) <= 1e-8, (tc, j)
            one = torch.zeros_like(fd[:1])
            P.ax_solve(op, fd[m - 1:].contiguous(), one, 1, 1e-8, 2000, P.AX_PCG_MIXED)
            assert np.array_equal(one[0].cpu().numpy(), un[m - 1]), tc
    finally:
        P.ax_destroy_operator(op)


# FP64 stencil with 4, 8 and 16 rows per CTA, cut at the last row and column.  The
# tolerance: some 12 roundings per node of terms that together are a few times the
# result for random data.
@pytest.mark.parametrize("nr,nz", [(1, 130), (3, 600), (4, 63), (333, 513), (1215, 40), (1217, 64), (2433, 129), (4900, 33)])
def test_fp64_stencil_rows_per_cta(nr, nz):
    op, ora, _, dev = _problem(nr, nz, 1)
    try:
        x = np.random.default_rng(nr).normal(size=(2, nr, nz))
        y = torch.zeros((2, nr, nz), dtype=torch.float64, device=dev)
        P.ax_apply_operator(op, torch.from_numpy(x).to(dev), y, 2)
        for j in range(2):
            ref = ora.apply_A(x[j])
            assert np.linalg.norm(y[j].cpu().numpy() - ref) <= 48 * 2.0 ** -53 * np.linalg.norm(ref)
    finally:
        P.ax_destroy_operator(op)
