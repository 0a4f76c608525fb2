"""Mixed solves of right-hand sides at both ends of the FP64 range.

The equations are linear and the mixed methods scale each right-hand side by a power
of two first, so a right-hand side 2^k f has the solution 2^k u bit for bit where no
entry of it overflows or is subnormal, and within one unit there.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1002_3094_gb300 as P  # noqa: E402
from paper_1002_3094_gb300.inputs import sample_operator_inputs  # noqa: E402
from workloads import layered_inclusion_medium  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart", [0, 1])
@pytest.mark.parametrize("method", [P.AX_PCG_MIXED, P.AX_CHEB_MIXED])
@pytest.mark.parametrize("guess", [False, True])
def test_scaled_right_hand_sides(method, guess, restart):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.load_library()
    nr, nz = 40, 50
    med = layered_inclusion_medium(n_rhs=1, nominal_n=64)
    kr, kz, q = sample_operator_inputs(med, nr, nz)
    # a source near r = 1, so that r f reaches 2^1023, in steps of 2^-30, so that 2^-1040 f is exact
    r, z = (np.arange(nr) + 0.5) / (nr + 0.5), (np.arange(nz) + 1) / (nz + 1.0)
    f = 0.99 * np.exp(-((r[:, None] - r[36]) ** 2 + (z[None, :] - z[20]) ** 2) / 0.005)
    f = np.round(f * 2.0 ** 30) * 2.0 ** -30
    ks = [0, 1024, 1023, 1022, 1000, -900] + ([] if guess else [-980])
    if method == P.AX_PCG_MIXED and not guess and not restart:
        ks.append(-1040)  # (the others round r f before the scaling)
    op = P.ax_setup_operator(*[torch.from_numpy(x).cuda() for x in (kr, kz, q)], nr, nz)
    try:
        P.ax_set_option(op, "mixed_restart", restart)
        fd = torch.from_numpy(np.stack([np.ldexp(f, k) for k in ks])).cuda()
        assert torch.isfinite(fd).all()
        u = torch.zeros_like(fd)
        flags = 0
        if guess:
            one = torch.zeros_like(fd[:1])
            P.ax_solve(op, fd[:1], one, 1, 1e-2, 1000, P.AX_PCG_MIXED)
            u = torch.from_numpy(np.stack([np.ldexp(one[0].cpu().numpy(), k) for k in ks])).cuda()
            flags = P.AX_FLAG_USE_GUESS
        st, info = P.ax_solve(op, fd, u, len(ks), 1e-9, 1000, method, flags)
        assert st == P.AX_OK
        got = u.cpu().numpy()
        assert np.abs(got[0]).max() < 1.0  # 2^k u does not overflow
        for j, k in enumerate(ks):
            assert info[j]["iters"] == info[0]["iters"]
            want = np.ldexp(got[0], k)
            ok = np.abs(want) >= 2.0 ** -1022
            assert np.array_equal(got[j][ok], want[ok]), k
            assert np.abs(got[j] - want).max() <= (0.0 if ok.all() else 2.0 ** -1074), k
    finally:
        P.ax_destroy_operator(op)
