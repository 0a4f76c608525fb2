"""FP64 mode solves against the same systems in extended precision.

T_l is an M-matrix whose smallest eigenvalue is some nr^2 times smaller than its
diagonal.  Factors formed without subtraction have a few roundings per row, so that the
solution is off by a few nr 2^-53, not by nr^2 2^-53; the tolerance is (nr + 8) 2^-53 of its
2-norm (roundings of random sign add up to less than their bound).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from paper_1002_3094_gb300.inputs import sample_operator_inputs  # noqa: E402
from workloads import layered_inclusion_medium  # noqa: E402

pytestmark = pytest.mark.gpu


def _solve_extended(f, kt, qt, bc_z):
    """Thomas in extended precision with the same subtraction-free pivots."""
    L = np.longdouble
    nr, nz = f.shape
    hr, hz = L(1.0 / (nr + 0.5)), L(1.0 / (nz if bc_z else nz + 1))
    lw = np.arange(nz).astype(L) + (0 if bc_z else 1)
    lam = 4 / hz ** 2 * np.sin(4 * np.arctan(L(1)) * lw / (2 * (nz if bc_z else nz + 1))) ** 2
    g = L(kt) * (np.arange(nr) + 1).astype(L) / hr
    ip, y, s = np.zeros((nr, nz), L), f.astype(L), 0
    for a in range(nr):
        s = (L(a) + L(0.5)) * hr * (L(kt) * lam + L(qt)) + (g[a - 1] * ip[a - 1] * s if a else 0)
        ip[a] = 1 / (g[a] + s)
        if a:
            y[a] += g[a - 1] * ip[a - 1] * y[a - 1]
    y[-1] *= ip[-1]
    for a in range(nr - 2, -1, -1):
        y[a] = (y[a] + g[a] * y[a + 1]) * ip[a]
    return y


# the register kernel with 8 and with 16 rows per lane, and the tall one
@pytest.mark.parametrize("nr,bc_z", [(2, 0), (65, 1), (333, 0), (500, 1), (1024, 0), (1024, 1), (1500, 1)])
def test_mode_solves(nr, bc_z):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    nz = 36
    med = layered_inclusion_medium(n_rhs=1, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz, bc_z=bc_z)
    f = np.random.default_rng(nr).normal(size=(1, nr, nz))
    op = P.ax_setup_operator(*[torch.from_numpy(x).cuda() for x in (kr, kz, q)], nr, nz, bc_z=bc_z)
    try:
        kt, qt = P.ax_operator_info(op)[:2]
        fd = torch.from_numpy(f).cuda()
        y = torch.zeros_like(fd)
        P.ax_apply_mode_solve(op, fd, y, 1)
        want = _solve_extended(f[0], kt, qt, bc_z)
        err = y[0].cpu().numpy() - want
        # by the column: the smooth modes dominate the whole
        assert (np.sqrt((err ** 2).sum(0)) <= (nr + 8) * 2.0 ** -53 * np.sqrt((want ** 2).sum(0))).all()
    finally:
        P.ax_destroy_operator(op)
