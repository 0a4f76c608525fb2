"""FP64 z-transforms by integer products at the ends of the FP64 range and of the
sizes they serve.

Tolerance as in test_gpu_digit_transform.py, 16 2^-53 of the row's 2-norm, and half a
unit of the smallest subnormal number, 2^-1075, for each of the n results.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from test_gpu_digit_transform import TOL, _matrix, _problem  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(op, x, nz, bc_z, dev):
    xl, mat = x.astype(np.longdouble), _matrix(nz, bc_z)
    norm = np.sqrt((xl ** 2).sum(1))
    for f, r in ((P.ax_apply_dst, mat.T), (P.ax_apply_dst_inverse, mat)):
        xd = torch.from_numpy(x).to(dev)
        y = torch.zeros_like(xd)
        f(op, xd, y, len(x))
        got = y.cpu().numpy()
        assert np.isfinite(got).all(), f.__name__
        err = np.sqrt(((got - xl @ r) ** 2).sum(1))
        assert (err <= TOL * norm + np.sqrt(nz) * np.ldexp(np.longdouble(1), -1075)).all(), (f.__name__, err / norm)


# rows whose largest entry has the exponent k or a little more, down to subnormal numbers
@pytest.mark.parametrize("nz,bc_z", [(128, 0), (300, 1)])
def test_rows_of_every_exponent(nz, bc_z):
    ks = [-1060, -1040, -1023, -1022, -1021, -1000, -950, -905, -901, -900, -899, -500, 0, 900, 1000, 1016]
    op, _, _, dev = _problem(48, nz, 1, bc_z)
    rng = np.random.default_rng(nz)
    x = np.ldexp(rng.normal(size=(48, nz)), np.resize(ks, 48)[:, None])
    try:
        _check(op, x, nz, bc_z, dev)
    finally:
        P.ax_destroy_operator(op)


@pytest.mark.parametrize("nz,bc_z", [(128, 0), (300, 1), (301, 1)])
def test_rows_near_the_largest_number(nz, bc_z):
    """Entries whose sums (the cosine transform folds its input) exceed the range, with
    transforms that do not."""
    op, _, _, dev = _problem(48, nz, 1, bc_z)
    big = 1.75 * 2.0 ** 1023
    x = np.zeros((48, nz))
    x[:, 5] = np.resize([big, -big, 0.5 * big], 48)
    x[::2, nz - 6] = big
    x[4:, 9] = np.ldexp(np.arange(44) - 21.5, 1010)
    x[40:, nz // 2] = 0.25 * big
    try:
        _check(op, x, nz, bc_z, dev)
    finally:
        P.ax_destroy_operator(op)
