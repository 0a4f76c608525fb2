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


@pytest.mark.parametrize("nz,bc_z", [(511, 1), (512, 0), (513, 1), (300, 0), (255, 1)])
def test_constant_rows(nz, bc_z):
    """Errors of the matrix entries that neighbours share would add up here.  Rounding P,
    Q and their sum costs at most 2 2^-53 of the row's norm, the entries' own rounding
    (2^-56 of the largest, of random sign) little: 3 2^-53."""
    rows = 64 if nz <= 512 else 384  # (fewer take the FFT above 512 columns)
    op, _, _, dev = _problem(64, nz, 1, bc_z)
    k = np.arange(nz)
    base = np.stack([np.ones(nz), np.where(k % 2, 1.0, -1.0), np.where(k < nz // 2, 1.0, 2.0), np.where(k % 7, 1.0, 3.0)])
    x = np.resize(base, (rows, nz))
    mat, xl = _matrix(nz, bc_z), x.astype(np.longdouble)
    try:
        for f, r in ((P.ax_apply_dst, mat.T), (P.ax_apply_dst_inverse, mat)):
            y = torch.zeros((rows, nz), dtype=torch.float64, device=dev)
            f(op, torch.from_numpy(x).to(dev), y, rows)
            err = np.sqrt(((y.cpu().numpy() - xl @ r) ** 2).sum(1) / (xl ** 2).sum(1))
            assert (err <= 3 * 2.0 ** -53).all(), (f.__name__, err[:4] * 2.0 ** 53)
    finally:
        P.ax_destroy_operator(op)
