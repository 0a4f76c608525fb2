"""FP64 z-transforms by integer products on the tensor cores.

Tolerance of the transforms, of the row's 2-norm: rounding the result costs at
most three half units (P, Q, their sum: 3 2^-53), rounding the input to 55 bits
below its largest entry sqrt(n) 2^-55 for a row with one large entry (n = 1024:
8 2^-53), the matrix and the products left out about 2^-53 each; 16 2^-53.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O  # noqa: E402
import paper_1002_3094_gb300 as P  # noqa: E402
from paper_1002_3094_gb300.inputs import sample_operator_inputs, sample_rhs  # noqa: E402
from workloads import layered_inclusion_medium  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 16 * 2.0 ** -53


def _problem(nr, nz, m, bc_z):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    med = layered_inclusion_medium(n_rhs=m, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz, bc_z=bc_z)
    dev = torch.device("cuda:0")
    op = P.ax_setup_operator(*[torch.from_numpy(x).to(dev) for x in (kr, kz, q)], nr, nz, bc_z=bc_z)
    return op, O.Operator(kr, kz, q, O.Grid(nr, nz, bc_z=bc_z)), sample_rhs(med, nr, nz, bc_z=bc_z), dev


def _matrix(n, bc_z):
    """The forward transform's matrix, angles reduced exactly."""
    L = np.longdouble
    pi, k = 4 * np.arctan(L(1)), np.arange(n)
    if bc_z == 0:
        return np.sqrt(L(2) / (n + 1)) * np.sin(pi * (np.outer(k + 1, k + 1) % (2 * n + 2)).astype(L) / (n + 1))
    c = np.sqrt(L(2) / n) * np.cos(pi * (np.outer(k, 2 * k + 1) % (4 * n)).astype(L) / (2 * n))
    c[0] *= np.sqrt(L(0.5))
    return c


# the smallest and largest sizes, K blocks of 32 and column tiles of 32 and 64 that end
# early or not at all, odd sizes, the smallest numbers of rows and row tiles of 128
@pytest.mark.parametrize("nz,rows,bc_z", [(128, 48, 0), (129, 127, 1), (130, 128, 0), (254, 129, 1), (511, 257, 0),
                                          (512, 50, 1), (641, 384, 1), (1023, 385, 0), (1023, 512, 1),
                                          (1024, 384, 0), (1024, 511, 1),
                                          (1024, 600, 0), (777, 641, 1)])  # (the last two: tiles of 64 columns)
def test_transform_against_extended_sums(nz, rows, bc_z):
    op, _, _, dev = _problem(rows, nz, 1, bc_z)
    rng = np.random.default_rng(nz + rows)
    base = rng.normal(size=(8, nz))
    base[1] = 0
    base[1, nz // 2] = 1.0
    base[2] *= np.exp(rng.uniform(-30, 30, nz))
    base[3] = 0
    base[4] = 1.0
    base[5] = np.sin(0.01 * np.arange(nz))
    base[6] = np.where(np.arange(nz) % 2, 1.0, -1.0) * (1 - 2.0 ** -53)  # every digit extreme
    scale = np.ldexp(1.0, rng.integers(-300, 300, rows))
    x = base[np.arange(rows) % 8] * scale[:, None]
    mat = _matrix(nz, bc_z)
    try:
        for f, r in ((P.ax_apply_dst, mat.T), (P.ax_apply_dst_inverse, mat)):
            ref = base.astype(np.longdouble) @ r
            norm = np.sqrt((base.astype(np.longdouble) ** 2).sum(1))
            xd = torch.from_numpy(x).to(dev)
            y = torch.zeros_like(xd)
            f(op, xd, y, rows)
            got = y.cpu().numpy() / scale[:, None]
            err = np.sqrt(((got - ref[np.arange(rows) % 8]) ** 2).sum(1).astype(float))
            assert (err <= TOL * norm[np.arange(rows) % 8]).all(), (f.__name__, err.max())
            f(op, xd, xd, rows)  # in place
            assert torch.equal(xd, y)
            # buffers that start 8 bytes off a 16-byte boundary
            flat_x, flat_y = (torch.zeros(rows * nz + 1, dtype=torch.float64, device=dev) for _ in range(2))
            flat_x[1:] = torch.from_numpy(x).to(dev).flatten()
            f(op, flat_x[1:].view(rows, nz), flat_y[1:].view(rows, nz), rows)
            assert torch.equal(flat_y[1:].view(rows, nz), y)
            # a row that is not finite stays alone
            xn = torch.from_numpy(x).to(dev)
            xn[3, 2], xn[17, nz - 1] = float("nan"), float("inf")
            f(op, xn, xn, rows)
            keep = [i for i in range(rows) if i not in (3, 17)]
            assert torch.equal(xn[keep], y[keep])
            assert not torch.isfinite(xn[[3, 17]]).any()
    finally:
        P.ax_destroy_operator(op)


@pytest.mark.parametrize("nr,nz,bc_z", [(48, 128, 0), (131, 257, 1), (70, 512, 0), (384, 1024, 0), (300, 511, 0), (400, 511, 1)])
def test_solves_meet_their_tolerance_alone_and_in_a_batch(nr, nz, bc_z):
    m = 3
    op, ora, f, dev = _problem(nr, nz, m, bc_z)
    fd = torch.from_numpy(f).to(dev)
    # the iteration stops on its own residual; the true one differs by some
    # (iterations) eps ||A|| ||u||, with ||A|| from the fastest oscillation
    v = np.where(np.add.outer(np.arange(nr), np.arange(nz)) % 2, -1.0, 1.0)
    norm_a = np.linalg.norm(ora.apply_A(v)) / np.linalg.norm(v)
    P.ax_set_option(op, "small_path", 0)  # else one small right-hand side takes a kernel without this transform
    try:
        for _ in range(4):  # launched directly, then as a captured graph
            u = torch.zeros_like(fd)
            st, info = P.ax_solve(op, fd, u, m, 1e-11, 2000, P.AX_PCG_FP64)
            assert st == P.AX_OK
            un = u.cpu().numpy()
            for j in range(m):
                phi = ora.phi(f[j])
                gap = info[j]["iters"] * 2.0 ** -52 * norm_a * np.linalg.norm(un[j])
                assert np.linalg.norm(phi - ora.apply_A(un[j])) <= 1e-11 * np.linalg.norm(phi) + gap
            one = torch.zeros_like(fd[:1])
            P.ax_solve(op, fd[m - 1:].contiguous(), one, 1, 1e-11, 2000, P.AX_PCG_FP64)
            assert torch.equal(one[0], u[m - 1])
    finally:
        P.ax_destroy_operator(op)


def test_an_expired_wait_shows_and_the_context_stays_usable():
    """The copy warp stops before its first block (a test option), the bounded
    waits run out: a solve returns AX_ERR_TIMEOUT, a transform NaN rows."""
    op, _, f, dev = _problem(64, 256, 1, 0)
    fd = torch.from_numpy(f).to(dev)
    x = torch.randn((64, 256), dtype=torch.float64, device=dev)
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    try:
        P.ax_set_option(op, "tc_stall_test", 1)
        P.ax_apply_dst(op, x, y, 64)
        assert torch.isnan(y).all()
        P.ax_apply_dst(op, x, y, 64)
        P.ax_apply_dst(op, y, z, 64)
        assert (z - x).norm() <= 2 * TOL * x.norm()
        P.ax_set_option(op, "small_path", 0)
        P.ax_set_option(op, "tc_stall_test", 1)
        with pytest.raises(P.AxError) as e:
            P.ax_solve(op, fd, torch.zeros_like(fd), 1, 1e-10, 50, P.AX_PCG_FP64)
        assert e.value.status == P.AX_ERR_TIMEOUT
        st, _ = P.ax_solve(op, fd, torch.zeros_like(fd), 1, 1e-10, 500, P.AX_PCG_FP64)
        assert st == P.AX_OK
    finally:
        P.ax_destroy_operator(op)
