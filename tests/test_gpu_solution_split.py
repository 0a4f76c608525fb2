"""The mode solves' operand by modes, read by the inverse tensor-core transform.

A preconditioner application with the mode-major kernel (14) against the staged one
(9), which writes the operand by rows, and against the FP64 one: rows that end
inside a lane's chunk, a piece of 8 and a block of 64 or 128, columns that end
inside a block of 8 positions, each chunk length (4, 8, 16 rows) and warp count.
Tolerances: the two do the same arithmetic up to the order of two additions (8
FP32 units of the largest intermediate, itself a few times the result); against
FP64 the transforms' 2^-16 twice and FP32 recurrences.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_1002_3094_gb300 as P  # noqa: E402
from paper_1002_3094_gb300.inputs import sample_operator_inputs  # noqa: E402
from workloads import layered_inclusion_medium  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc_z", [0, 1])
@pytest.mark.parametrize("nr,nz", [(3, 2), (63, 17), (65, 130), (129, 7), (250, 127), (257, 64), (511, 33), (513, 258),
                                   (777, 100), (1023, 31), (1025, 140), (2047, 19), (2049, 130), (4095, 23), (4096, 9)])
def test_by_modes_against_by_rows(nr, nz, bc_z):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    m = 2
    dev = torch.device("cuda:0")
    med = layered_inclusion_medium(n_rhs=m, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz, bc_z=bc_z)
    op = P.ax_setup_operator(*[torch.from_numpy(x).to(dev) for x in (kr, kz, q)], nr, nz, bc_z=bc_z)
    try:
        x = torch.from_numpy(np.random.default_rng(nr + nz).normal(size=(m, nr, nz))).to(dev)
        ref, out = torch.zeros_like(x), {}
        P.ax_apply_preconditioner(op, x, ref, m)
        P.ax_set_option(op, "dst_tensor", 1)
        for kernel in (9, 14):
            P.ax_set_option(op, "mode_kernel", kernel)
            out[kernel] = torch.zeros_like(x)
            P.ax_apply_preconditioner(op, x, out[kernel], m, P.AX_PREC_FP32_TC3)
        for j in range(m):
            assert (out[14][j] - out[9][j]).norm() <= 2.0 ** -19 * ref[j].norm()
            assert (out[14][j] - ref[j]).norm() <= 2.0 ** -13 * ref[j].norm()
        # a right-hand side that is not finite leaves nothing behind in the padding
        bad = x.clone()
        bad[0, nr // 2, nz // 2] = float("nan")
        again = torch.zeros_like(x)
        P.ax_apply_preconditioner(op, bad, again, m, P.AX_PREC_FP32_TC3)
        assert torch.equal(again[1], out[14][1])
        P.ax_apply_preconditioner(op, x, again, m, P.AX_PREC_FP32_TC3)
        assert torch.equal(again, out[14])
    finally:
        P.ax_destroy_operator(op)


@pytest.mark.parametrize("bc_z", [0, 1])
@pytest.mark.parametrize("nr,nz", [(1, 5), (7, 3), (8, 4), (9, 6), (63, 9), (65, 7), (449, 2), (511, 5), (512, 4),
                                   (513, 5), (897, 1), (1023, 6), (1024, 3), (1025, 2)])
def test_fp64_mode_solves_at_chunk_edges(nr, nz, bc_z):
    """Backward error of every mode system where rows end at the edge of a chunk (8
    or 16 rows), a warp (8 chunks) and the kernel's range, columns inside a CTA's 4:
    the recurrences round each row a few times, 1e-14 as a stable solver."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    m = 2
    dev = torch.device("cuda:0")
    med = layered_inclusion_medium(n_rhs=m, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz, bc_z=bc_z)
    grid = O.Grid(nr, nz, bc_z=bc_z)
    kt, qt = O.preconditioner_constants(kr, kz, q)[:2]
    op = P.ax_setup_operator(*[torch.from_numpy(x).to(dev) for x in (kr, kz, q)], nr, nz, bc_z=bc_z)
    try:
        b = np.random.default_rng(nr).normal(size=(m, nr, nz))
        y = torch.zeros((m, nr, nz), dtype=torch.float64, device=dev)
        P.ax_apply_mode_solve(op, torch.from_numpy(b).to(dev), y, m)
        y = y.cpu().numpy()
        lam = O.mode_eigenvalues(nz, grid.hz, bc_z)
        for l in range(nz):
            sub, diag, sup = O.mode_tridiagonal(kt, qt, lam[l], grid)
            t = np.diag(diag) + (np.diag(sub, -1) + np.diag(sup, 1) if nr > 1 else 0.0)
            norm = np.abs(t).sum(1).max()
            for j in range(m):
                r = t @ y[j, :, l] - b[j, :, l]
                assert np.linalg.norm(r) <= 1e-14 * (norm * np.linalg.norm(y[j, :, l]) + np.linalg.norm(b[j, :, l]))
    finally:
        P.ax_destroy_operator(op)
