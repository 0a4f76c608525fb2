"""The work that users of the solver have it do, as cases that can be timed.

A case is a dict of plain values; ``prepare`` makes what a program holds before
the call (the medium's operator, the right-hand sides, the network), ``run`` is
one pass through the public entry points, ``exact`` the same result in 64 bits
from plain torch.  The kinds:

  solve      ax_solve on a set-up operator: many (or one) right-hand sides of
             one medium, each method and z boundary
  medium     a medium that is used once: set up, solve, destroy (how training
             sets and parameter studies call the library)
  chain      Laguerre harmonics: sequential warm-started solves, each
             right-hand side formed from the solutions before it
  batch      independent operators of uneven grid sizes in one call
  precond    one preconditioner application, for a caller's own Krylov method
  guess      inference of the initial-guess network
  gradients  loss and gradients of the initial-guess network

Media are the benchmark's kinds: smooth bumps, z-layers with inclusions and
random fields; sources are Gaussians.  Mixed-precision and Chebyshev solves
run to 1e-10, the tolerance at which the paper counts its iterations, and
grids above 2048 x 2048 to 1e-9.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1002_3094_gb300 as P
from paper_1002_3094_gb300.inputs import sample_points
from paper_1002_3094_gb300.laguerre import solve_chain

ALPHA = 5                      # Laguerre order of the chain
SIZES = (127, 255, 511, 1023)  # grid sizes of the uneven batch
CHANNELS = (24, 48, 96, 192)   # the network's default channels
MAX_ITER = 20000


def listed():
    return [
        # the smallest call: one source on a 64 x 64 grid, plain FP64 (latency)
        dict(name="solve_64_fp64", kind="solve", nr=64, nz=64, m=1, bc_z=0, method="pcg64", medium="bumps", tol=1e-10),
        # one random-field medium, used once: set-up, one mixed solve, destroy
        dict(name="medium_256_mixed", kind="medium", nr=256, nz=256, m=1, bc_z=0, method="pcg_mixed", medium="field",
             tol=1e-10),
        # a stretch of the Laguerre chain: one right-hand side at a time, zero-flux z
        dict(name="chain_1024_zero_flux", kind="chain", nr=1024, nz=1024, harmonics=4, bc_z=1, tol=1e-10),
        # the benchmark: 64 point sources in one layered medium
        dict(name="solve_1024_m64_mixed", kind="solve", nr=1024, nz=1024, m=64, bc_z=0, method="pcg_mixed",
             medium="layers", tol=1e-10),
        # a ragged grid with the zero-flux boundary, a moderate number of sources
        dict(name="solve_777x1000_m24_zero_flux", kind="solve", nr=777, nz=1000, m=24, bc_z=1, method="pcg_mixed",
             medium="layers", tol=1e-10),
        # the largest: 16 sources on a 4096 x 4096 grid
        dict(name="solve_4096_m16_mixed", kind="solve", nr=4096, nz=4096, m=16, bc_z=0, method="pcg_mixed",
             medium="layers", tol=1e-9),
        # many media of uneven sizes at once
        dict(name="batch_24_uneven", kind="batch", count=24, bc_z=0, tol=1e-10),
        # plain FP64 with several right-hand sides
        dict(name="solve_500x511_m8_fp64", kind="solve", nr=500, nz=511, m=8, bc_z=0, method="pcg64", medium="layers",
             tol=1e-10),
        # Chebyshev (no inner products), mixed precision
        dict(name="solve_511_m16_cheb_mixed", kind="solve", nr=511, nz=511, m=16, bc_z=0, method="cheb_mixed",
             medium="field", tol=1e-10),
        # the preconditioner alone in FP64, inside a caller's own iteration
        dict(name="precond_1024_m8_fp64", kind="precond", nr=1024, nz=1024, m=8, bc_z=0, medium="layers"),
        # initial-guess network: inference for a batch of 256 x 256 media
        dict(name="guess_256_b16", kind="guess", hw=256, batch=16),
        # initial-guess network: a training batch
        dict(name="gradients_256_b16", kind="gradients", hw=256, batch=16, h1=10.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, m_max, unknowns):
    """Grid and right-hand sides, log-uniform, at most `unknowns` in all."""
    while True:
        nr, nz, m = _log_int(rng, lo, hi), _log_int(rng, lo, hi), _log_int(rng, 1, m_max)
        if nr * nz * m <= unknowns:
            return nr, nz, m


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "medium", "chain", "batch", "precond", "guess",
                       "gradients"])
    bc_z = rng.randrange(2)
    if kind == "solve":
        method = rng.choice(["pcg_mixed", "pcg_mixed", "pcg_mixed", "pcg64", "cheb_mixed"])
        if method == "pcg_mixed":
            nr, nz, m = _grid(rng, 48, 4096, 64, 1 << 26)
        elif method == "pcg64":
            nr, nz, m = _grid(rng, 32, 1024, 8, 1 << 22)
        else:
            nr, nz, m = _grid(rng, 64, 1024, 32, 1 << 23)
        medium = rng.choice({"pcg_mixed": ["layers", "field"], "pcg64": ["layers", "bumps"],
                             "cheb_mixed": ["field", "layers"]}[method])
        return dict(kind=kind, nr=nr, nz=nz, m=m, bc_z=bc_z, method=method, medium=medium,
                    tol=1e-10 if max(nr, nz) <= 2048 else 1e-9)
    if kind == "medium":
        nr, nz, m = _grid(rng, 64, 1024, 4, 1 << 21)
        return dict(kind=kind, nr=nr, nz=nz, m=m, bc_z=bc_z, method="pcg_mixed",
                    medium=rng.choice(["field", "layers"]), tol=1e-10)
    if kind == "chain":
        nr, nz, _ = _grid(rng, 128, 2048, 1, 1 << 21)
        return dict(kind=kind, nr=nr, nz=nz, harmonics=rng.randrange(2, 7), bc_z=1, tol=1e-10)
    if kind == "batch":
        return dict(kind=kind, count=rng.randrange(4, 33), bc_z=bc_z, tol=1e-10)
    if kind == "precond":
        nr, nz, m = _grid(rng, 64, 2048, 16, 1 << 24)
        return dict(kind=kind, nr=nr, nz=nz, m=m, bc_z=bc_z, medium="layers")
    hw = 8 * _log_int(rng, 4, 40)
    batch = rng.randrange(1, max(2, min(32, (1 << 20) // (hw * hw)) + 1))
    return dict(kind=kind, hw=hw, batch=batch) if kind == "guess" else dict(kind=kind, hw=hw, batch=batch,
                                                                            h1=rng.choice([0.0, 10.0]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dev(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def _kappa(rng, medium, n, max_contrast=10.0):
    """A function kappa(r, z) of device vectors (FP64 [len(r)][len(z)])."""
    if medium == "bumps":
        amps, centres = rng.uniform(0.0, 2.0, 3), rng.uniform(0.0, 1.0, (3, 2))

        def f(r, z):
            out = torch.ones((r.numel(), z.numel()), dtype=torch.float64, device="cuda")
            for a, (rc, zc) in zip(amps, centres):
                out += a * torch.exp(-((r[:, None] - rc) ** 2 + (z[None, :] - zc) ** 2) / 0.02)
            return out
        return f
    if medium == "layers":
        cuts, values = np.sort(rng.uniform(0.0, 1.0, 7)), max_contrast ** rng.uniform(0.0, 1.0, 8)
        rc, zc = rng.uniform(0.2, 0.8, 2)
        a, b = rng.uniform(0.05, 0.2, 2)
        width = 2.0 / n

        def f(r, z):
            lay = _dev(values)[torch.searchsorted(_dev(cuts), z, right=True)]
            rho = torch.sqrt(((r[:, None] - rc) / a) ** 2 + ((z[None, :] - zc) / b) ** 2)
            inc = 0.5 * (1.0 - torch.tanh(0.5 * (rho - 1.0) * min(a, b) / width))
            return lay[None, :] * (1.0 + 4.0 * inc)
        return f
    om, ph = rng.normal(0.0, 10.0, (64, 2)), rng.uniform(0.0, 2.0 * np.pi, 64)
    contrast = rng.uniform(2.0, 10.0)

    def f(r, z):  # noqa: F811
        # cos(w1 r + w2 z + phi) as a sum of products: two small GEMMs
        ar, az = torch.outer(r, _dev(om[:, 0])), torch.outer(z, _dev(om[:, 1])) + _dev(ph)
        g = torch.cos(ar) @ torch.cos(az).T - torch.sin(ar) @ torch.sin(az).T
        t = ((g / math.sqrt(32.0) + 2.5) / 5.0).clamp(0.0, 1.0)
        return torch.exp(math.log(contrast) * t)
    return f


def _medium(rng, medium, nr, nz, bc_z):
    """kappa_r, kappa_z, q at the grid's sample points (FP64, on the GPU)."""
    rn, rf, zn, zf = (_dev(a) for a in sample_points(nr, nz, bc_z=bc_z))
    kappa = _kappa(rng, medium, min(nr, nz))
    kr, kz = kappa(rf, zn).contiguous(), kappa(rn, zf).contiguous()
    if medium == "bumps":
        q = torch.full((nr, nz), 0.1, dtype=torch.float64, device="cuda")
    elif medium == "layers":
        k = kappa(rn, zn)
        q = (5.0 / torch.exp(torch.log(k).mean()) * k).contiguous()
    else:
        q = torch.full((nr, nz), float(rng.uniform(0.05, 0.5)), dtype=torch.float64, device="cuda")
    return kr, kz, q


def _sources(rng, medium, nr, nz, m, bc_z):
    """Gaussian sources: of width 0.05 for the bumps, else point-like (two grid spacings)."""
    rn, _, zn, _ = (_dev(a) for a in sample_points(nr, nz, bc_z=bc_z))
    sr, sz = (0.05, 0.05) if medium == "bumps" else (2.0 / nr, 2.0 / nz)
    f = torch.empty((m, nr, nz), dtype=torch.float64, device="cuda")
    for j in range(m):
        rc, zc = rng.uniform(0.05, 0.95, 2)
        f[j] = torch.outer(torch.exp(-(rn - rc) ** 2 / (2 * sr * sr)), torch.exp(-(zn - zc) ** 2 / (2 * sz * sz)))
    return f


def _problem(case, seed):
    rng = np.random.default_rng([seed, case["nr"], case["nz"]])
    nr, nz, bc_z = case["nr"], case["nz"], case["bc_z"]
    med = _medium(rng, case["medium"], nr, nz, bc_z)
    return med, _sources(rng, case["medium"], nr, nz, case["m"], bc_z)


def _chain_problem(case, seed):
    rng = np.random.default_rng([seed, case["nr"], case["nz"], 7])
    nr, nz = case["nr"], case["nz"]
    rn, rf, zn, zf = (_dev(a) for a in sample_points(nr, nz, bc_z=1))
    # four layers of rising squared wave speed; q = h^2 / 4 in units of the domain
    cuts, v2 = np.sort(rng.uniform(0.15, 0.85, 3)), np.sort(rng.uniform(1.0, 5.0, 4))
    lay = lambda z: _dev(v2)[torch.searchsorted(_dev(cuts), z, right=True)][None, :]  # noqa: E731
    kr, kz = lay(zn).expand(nr, nz).contiguous(), lay(zf).expand(nr, nz + 1).contiguous()
    q = torch.full((nr, nz), 1.0e4, dtype=torch.float64, device="cuda")
    sg = 4.0 / min(nr, nz)
    src = torch.outer(torch.exp(-rn ** 2 / (2 * sg * sg)), torch.exp(-(zn - 0.3) ** 2 / (2 * sg * sg)))
    fm = rng.uniform(0.5, 1.0, case["harmonics"]) * np.where(rng.uniform(size=case["harmonics"]) < 0.5, -1.0, 1.0)
    return (kr, kz, q), 4.0 * q, src, [float(x) for x in fm]


def _batch_problem(case, seed):
    rng = np.random.default_rng([seed, case["count"], 3])
    out = []
    for j in range(case["count"]):
        # the sizes belong to the case, the media to the seed
        nr, nz = SIZES[(j * 7 + case["count"]) % 4], SIZES[(j * 5 + j // 4) % 4]
        med = _medium(rng, "layers" if j % 3 else "field", nr, nz, case["bc_z"])
        out.append((nr, nz, med, _sources(rng, "field", nr, nz, 1, case["bc_z"])[0]))
    return out


def _layers_of_net():
    c1, c2, c3, c4 = CHANNELS
    return [(3, c1), (c1, c1), (c1, c2), (c2, c2), (c2, c3), (c3, c3), (c3, c4), (c4, c4), (c4, c3), (c3, c3),
            (c3, c2), (c2, c2), (c2, c1), (c1, c1)]


def _net_problem(case, seed):
    """Flat parameters (He-normal weights, small biases), features and targets."""
    rng = np.random.default_rng([seed, case["hw"], case["batch"], 11])
    flat = []
    for cin, cout in _layers_of_net():
        flat += [rng.normal(0.0, math.sqrt(2.0 / (9 * cin)), 9 * cin * cout), rng.normal(0.0, 0.05, cout)]
    flat += [rng.normal(0.0, math.sqrt(1.0 / CHANNELS[0]), CHANNELS[0]), rng.normal(0.0, 0.05, 1)]
    hw, b = case["hw"], case["batch"]
    gen = torch.Generator("cuda").manual_seed(seed)
    # smooth features: random low-resolution fields, interpolated
    low = torch.randn((b, 3, 16, 16), generator=gen, device="cuda")
    x = torch.nn.functional.interpolate(low, size=(hw, hw), mode="bilinear", align_corners=False).contiguous()
    low = torch.randn((b, 1, 16, 16), generator=gen, device="cuda")
    t = torch.nn.functional.interpolate(low, size=(hw, hw), mode="bilinear", align_corners=False)[:, 0].contiguous()
    return np.concatenate(flat).astype(np.float32), x, t


class _Handle:
    """Owns a library object until the state is dropped."""

    def __init__(self, value, destroy):
        self.value, self._destroy = value, destroy

    def __del__(self):
        self._destroy(self.value)


def _operator(med, nr, nz, bc_z):
    return _Handle(P.ax_setup_operator(*med, nr, nz, bc_z=bc_z), P.ax_destroy_operator)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "precond"):
        med, f = _problem(case, seed)
        if kind == "precond":
            gen = torch.Generator("cuda").manual_seed(seed)
            f = torch.randn(f.shape, generator=gen, device="cuda", dtype=torch.float64)
        return dict(case=case, op=_operator(med, case["nr"], case["nz"], case["bc_z"]), f=f, u=torch.zeros_like(f))
    if kind == "medium":
        med, f = _problem(case, seed)
        return dict(case=case, med=med, f=f, u=torch.zeros_like(f))
    if kind == "chain":
        med, c2, src, fm = _chain_problem(case, seed)
        nr, nz = case["nr"], case["nz"]
        return dict(case=case, op=_operator(med, nr, nz, 1), c2=c2, src=src, fm=fm,
                    q=torch.zeros((1, nr, nz), dtype=torch.float64, device="cuda"),
                    work=torch.zeros((3, nr, nz), dtype=torch.float64, device="cuda"))
    if kind == "batch":
        items = _batch_problem(case, seed)
        ops = [_operator(med, nr, nz, case["bc_z"]) for nr, nz, med, _ in items]
        batch = _Handle(P.ax_batch_create([o.value for o in ops]), P.ax_batch_destroy)
        return dict(case=case, batch=batch, fs=[f.contiguous() for *_, f in items],
                    us=[torch.zeros_like(f) for *_, f in items])
    flat, x, t = _net_problem(case, seed)
    net = _Handle(P.ax_guessnet_create(case["hw"], CHANNELS, batch_capacity=case["batch"], seed=1),
                  P.ax_guessnet_destroy)
    P.ax_guessnet_set_params(net.value, flat)
    if kind == "gradients":
        P.ax_guessnet_set_loss(net.value, case["h1"])
    return dict(case=case, net=net, x=x, t=t, y=torch.zeros_like(t))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        P.ax_solve(state["op"].value, state["f"], state["u"], case["m"], case["tol"], MAX_ITER,
                   P.METHODS[case["method"]])
        return state["u"]
    if kind == "medium":
        op = P.ax_setup_operator(*state["med"], case["nr"], case["nz"], bc_z=case["bc_z"])
        P.ax_solve(op, state["f"], state["u"], case["m"], case["tol"], MAX_ITER, P.METHODS[case["method"]])
        P.ax_destroy_operator(op)
        return state["u"]
    if kind == "chain":
        solve_chain(state["op"].value, state["c2"], state["src"], state["fm"], ALPHA, case["tol"], state["q"],
                    state["work"])
        return {"last": state["q"], "fields": state["work"]}
    if kind == "batch":
        P.ax_batch_solve(state["batch"].value, state["fs"], state["us"], case["tol"], MAX_ITER, P.AX_PCG_MIXED)
        return state["us"]
    if kind == "precond":
        P.ax_apply_preconditioner(state["op"].value, state["f"], state["u"], case["m"], P.AX_PREC_FP64)
        return state["u"]
    if kind == "guess":
        P.ax_guessnet_forward(state["net"].value, state["x"], state["y"], case["batch"])
        return state["y"]
    loss, grad = P.ax_guessnet_gradients(state["net"].value, state["x"], state["t"], case["batch"])
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------------------
# work: inputs read once, outputs written once; the arithmetic of a nominal
# number of iterations (stencil, vector updates, two fast transforms and the
# tridiagonal solves)
# ---------------------------------------------------------------------------
NOMINAL_ITERATIONS = 30


def _iteration_flops(nr, nz):
    return nr * nz * (30 + 2 * 5 * math.log2(2 * nz))


def work(case):
    kind = case["kind"]
    if kind in ("solve", "medium"):
        n = case["nr"] * case["nz"]
        return dict(bytes=16 * n * case["m"] + 24 * n,
                    flops=NOMINAL_ITERATIONS * case["m"] * _iteration_flops(case["nr"], case["nz"]))
    if kind == "chain":
        n = case["nr"] * case["nz"]
        return dict(bytes=8 * (3 + 2 + 4) * n,
                    flops=NOMINAL_ITERATIONS * case["harmonics"] * _iteration_flops(case["nr"], case["nz"]))
    if kind == "batch":
        grids = [(SIZES[(j * 7 + case["count"]) % 4], SIZES[(j * 5 + j // 4) % 4]) for j in range(case["count"])]
        return dict(bytes=sum(40 * a * b for a, b in grids),
                    flops=NOMINAL_ITERATIONS * sum(_iteration_flops(a, b) for a, b in grids))
    if kind == "precond":
        n = case["nr"] * case["nz"]
        return dict(bytes=16 * n * case["m"] + 8 * n,
                    flops=case["m"] * n * (10 + 2 * 5 * math.log2(2 * case["nz"])))
    res = [1, 1, 2, 2, 4, 4, 8, 8, 4, 4, 2, 2, 1, 1]  # down-sampling of each layer
    plane = case["hw"] ** 2 * case["batch"]
    flops = sum(18.0 * a * b * plane / (d * d) for (a, b), d in zip(_layers_of_net(), res))
    params = sum(9 * a * b + b for a, b in _layers_of_net())
    if kind == "guess":
        return dict(bytes=16 * plane + 4 * params, flops=flops)
    return dict(bytes=16 * plane + 8 * params, flops=3 * flops)


# ---------------------------------------------------------------------------
# 64-bit results
# ---------------------------------------------------------------------------
class _Exact:
    """The discrete operator and its preconditioner in plain FP64 torch."""

    def __init__(self, kr, kz, q, nr, nz, bc_z):
        rn, rf, _, _ = (_dev(a) for a in sample_points(nr, nz, bc_z=bc_z))
        hr, hz = 1.0 / (nr + 0.5), 1.0 / (nz if bc_z else nz + 1)
        self.nr, self.nz, self.bc = nr, nz, bc_z
        self.r = rn
        self.cr = rf[:, None] * kr / hr ** 2
        self.cz = rn[:, None] * kz / hz ** 2
        if bc_z:
            self.cz[:, 0] = 0.0
            self.cz[:, -1] = 0.0
        self.w = rn[:, None] * q
        kt = 0.5 * (min(kr.min(), kz.min()) + max(kr.max(), kz.max()))
        qt = 0.5 * (q.min() + q.max())
        ll = torch.arange(nz, device="cuda", dtype=torch.float64) + (0.0 if bc_z else 1.0)
        self.angle = math.pi * ll / (2.0 * (nz if bc_z else nz + 1))
        lam = 4.0 / hz ** 2 * torch.sin(self.angle) ** 2
        e = -kt * rf / hr ** 2
        d = kt * ((rf + torch.cat([rf.new_zeros(1), rf[:-1]])) / hr ** 2)[:, None] + rn[:, None] * (kt * lam + qt)
        self.e = e[:-1]
        self.ip = torch.empty_like(d)  # inverse Thomas pivots
        self.ip[0] = 1.0 / d[0]
        for i in range(1, nr):
            self.ip[i] = 1.0 / (d[i] - self.e[i - 1] ** 2 * self.ip[i - 1])

    def apply(self, y):
        out = self.w * y
        dr = self.cr[:-1] * (y[:, :-1] - y[:, 1:])
        out[:, :-1] += dr
        out[:, 1:] -= dr
        out[:, -1] += self.cr[-1] * y[:, -1]
        dz = self.cz[:, 1:-1] * (y[..., :-1] - y[..., 1:])
        out[..., :-1] += dz
        out[..., 1:] -= dz
        out[..., 0] += self.cz[:, 0] * y[..., 0]
        out[..., -1] += self.cz[:, -1] * y[..., -1]
        return out

    def _sine(self, x):
        z = x.new_zeros(x.shape[:-1] + (1,))
        ext = torch.cat([z, x, z, -x.flip(-1)], dim=-1)
        return -torch.fft.rfft(ext).imag[..., 1:self.nz + 1] * math.sqrt(0.5 / (self.nz + 1))

    def _cos(self, x):
        t = torch.fft.rfft(torch.cat([x, x.flip(-1)], dim=-1))[..., :self.nz]
        out = (t.real * torch.cos(self.angle) + t.imag * torch.sin(self.angle)) * math.sqrt(0.5 / self.nz)
        out[..., 0] *= math.sqrt(0.5)
        return out

    def _cos_inverse(self, x):
        x = x.clone()
        x[..., 0] *= math.sqrt(2.0)
        spec = torch.complex(x * torch.cos(self.angle), x * torch.sin(self.angle))
        spec = torch.cat([spec, spec.new_zeros(spec.shape[:-1] + (1,))], dim=-1)
        return torch.fft.irfft(spec, n=2 * self.nz)[..., :self.nz] * math.sqrt(2.0 * self.nz)

    def precond(self, v):
        t = (self._cos(v) if self.bc else self._sine(v)).transpose(0, 1).contiguous()  # [nr][m][nz]
        ip, e = self.ip, self.e.tolist()
        for i in range(1, self.nr):
            t[i] -= (e[i - 1] * ip[i - 1]) * t[i - 1]
        t[-1] *= ip[-1]
        for i in range(self.nr - 2, -1, -1):
            t[i] = (t[i] - e[i] * t[i + 1]) * ip[i]
        t = t.transpose(0, 1)
        return self._cos_inverse(t) if self.bc else self._sine(t.contiguous())

    def solve(self, f):
        """PCG to a relative residual of 1e-14, once restarted from the true residual."""
        phi = self.r[:, None] * f
        bb = phi.square().sum(dim=(1, 2), keepdim=True)
        x = torch.zeros_like(phi)
        for _ in range(2):
            r = phi - self.apply(x)
            z = self.precond(r)
            p, rho = z, (r * z).sum(dim=(1, 2), keepdim=True)
            for it in range(400):
                q = self.apply(p)
                alpha = rho / (p * q).sum(dim=(1, 2), keepdim=True).clamp_min(1e-300)
                x = x + alpha * p
                r = r - alpha * q
                if it % 4 == 3 and bool((r.square().sum(dim=(1, 2), keepdim=True) <= 1e-28 * bb).all()):
                    break
                z = self.precond(r)
                new = (r * z).sum(dim=(1, 2), keepdim=True)
                p = z + (new / rho.clamp_min(1e-300)) * p
                rho = new
        return x


def _net_exact(case, flat, x, t):
    p = torch.tensor(flat, dtype=torch.float64, device="cuda", requires_grad=case["kind"] == "gradients")
    off = 0

    def conv(a, cin, cout):
        nonlocal off
        w = p[off:off + 9 * cin * cout].view(3, 3, cin, cout).permute(3, 2, 0, 1)
        off += 9 * cin * cout
        b = p[off:off + cout]
        off += cout
        # im2col and a product: plain FP64
        cols = torch.nn.functional.unfold(a, 3, padding=1)
        y = (w.reshape(cout, -1) @ cols).view(a.shape[0], cout, *a.shape[2:]) + b[None, :, None, None]
        return torch.relu(y)

    pool, up = (lambda a: torch.nn.functional.avg_pool2d(a, 2)), (lambda a: torch.nn.functional.interpolate(
        a, scale_factor=2, mode="nearest"))
    c1, c2, c3, c4 = CHANNELS
    a = x.double()
    s1 = conv(conv(a, 3, c1), c1, c1)
    s2 = conv(conv(pool(s1), c1, c2), c2, c2)
    s3 = conv(conv(pool(s2), c2, c3), c3, c3)
    b = conv(conv(pool(s3), c3, c4), c4, c4)
    d = conv(conv(up(b), c4, c3) + s3, c3, c3)
    d = conv(conv(up(d), c3, c2) + s2, c2, c2)
    d = conv(conv(up(d), c2, c1) + s1, c1, c1)
    y = (d * p[off:off + c1][None, :, None, None]).sum(1) + p[off + c1]
    if case["kind"] == "guess":
        return y
    e = y - t.double()
    loss = e.square().sum() + case["h1"] * ((e[:, 1:] - e[:, :-1]).square().sum()
                                            + (e[:, :, 1:] - e[:, :, :-1]).square().sum())
    loss = loss / e.numel()
    return loss, torch.autograd.grad(loss, p)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "medium"):
        n = case["nr"] * case["nz"] * case["m"]
        if n > 1 << 26 or case["nr"] > 2048:
            return None
        med, f = _problem(case, seed)
        return _Exact(*med, case["nr"], case["nz"], case["bc_z"]).solve(f)
    if kind == "precond":
        med, f = _problem(case, seed)
        gen = torch.Generator("cuda").manual_seed(seed)
        f = torch.randn(f.shape, generator=gen, device="cuda", dtype=torch.float64)
        return _Exact(*med, case["nr"], case["nz"], case["bc_z"]).precond(f)
    if kind == "batch":
        out = []
        for j, (nr, nz, med, f) in enumerate(_batch_problem(case, seed)):
            out.append(_Exact(*med, nr, nz, case["bc_z"]).solve(f[None])[0] if j < 8 else None)
        return out
    if kind == "chain":
        med, c2, src, fm = _chain_problem(case, seed)
        ex = _Exact(*med, case["nr"], case["nz"], 1)
        big_t, big_s = torch.zeros_like(src), torch.zeros_like(src)
        f = fm[0] * src
        for k in range(len(fm)):
            sol = ex.solve(f[None])
            if k + 1 < len(fm):
                big_t = big_t + _weights(k)[1] * sol[0]
                big_s = big_s + big_t
                f = fm[k + 1] * src - c2 * _weights(k + 1)[0] * big_s
        return {"last": sol, "fields": torch.stack([big_t, big_s, f])}
    flat, x, t = _net_problem(case, seed)
    # a sample at a time bounds the memory of the unfolded inputs
    if kind == "guess":
        with torch.no_grad():
            return torch.cat([_net_exact(case, flat, x[i:i + 1], t[i:i + 1]) for i in range(case["batch"])])
    parts = [_net_exact(case, flat, x[i:i + 1], t[i:i + 1]) for i in range(case["batch"])]
    return {"loss": float(sum(a for a, _ in parts)) / len(parts),
            "grad": (sum(g for _, g in parts) / len(parts)).cpu().numpy()}


def _weights(m):
    """(sqrt(m! / (m + alpha)!), sqrt((m + alpha)! / m!)) from the factorials."""
    w = math.sqrt(math.factorial(m + ALPHA) / math.factorial(m))
    return 1.0 / w, w
