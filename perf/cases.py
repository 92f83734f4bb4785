"""Workloads of the TENO-AA library for timing and for comparing builds.

Each case goes through the public entry points (paper_2109_14340_gb300) the
way a solver program does.  Kinds of pass:

  rhs      one right-hand side of a state, optionally with its decision record
  steps    load the state, then per step the CFL time step and one SSP-RK3 step
  batch    load every problem's state, then graph-captured steps of the batch
  rollout  differentiable run: final state and the gradient of a density
           mismatch with respect to the initial state

The states are the ones a run meets after its first steps: interfaces a few
cells wide, plateaus that differ by rounding only, resolved smooth waves.
`exact` evaluates the same formulas in plain FP64 PyTorch (Fu, arXiv
2109.14340: Sec. 3-5 and App. A), written for whole arrays and sharing nothing
with the library.
"""
import functools
import math
from fractions import Fraction

import torch
import torch.utils.checkpoint

import paper_2109_14340_gb300 as T

PERIODIC, TRANSMISSIVE, SLIP, NOSLIP, DIRICHLET = 0, 1, 2, 3, 4
DEV = "cuda"
F64 = torch.float64


def _grid(name, kind, field, n, scheme, **kw):
    n = list(n) + [1] * (3 - len(n))
    c = dict(kind=kind, field=field, nx=n[0], ny=n[1], nz=n[2], scheme=scheme, steps=1, every=1,
             record=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _batch(name, count, nmin, nmax, steps):
    c = dict(kind="batch", field="batch", count=count, nmin=nmin, nmax=nmax, steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one right-hand side of the 400-cell shock tube, called from a user's
        # own time integrator: the smallest call, all launch and latency
        _grid("rhs_1d_400", "rhs", "tube", [400], 8),
        # the 400-cell shock tube advanced by the library itself
        _grid("tube_1d_400", "steps", "tube", [400], 8, steps=10),
        # a small 2D run, far too few faces to fill the GPU
        _grid("quadrants_2d_128", "steps", "quadrants", [128, 128], 10, steps=4),
        # a long and thin ragged grid with walls, twelve-point scheme, right-hand
        # side with its decision record (diagnostics, recording runs)
        _grid("walls_2d_record", "rhs", "walls", [509, 203], 12, record=True),
        # the 2D four-quadrant problem at its full size
        _grid("quadrants_2d_1024", "steps", "quadrants", [1024, 1024], 10),
        # 3D turbulence at the size of a parameter study
        _grid("turbulence_3d_64", "steps", "turbulence", [64, 64, 64], 10, steps=2),
        # 3D implosion with limiter, Rusanov splitting, walls and Dirichlet inflow
        _grid("noh_3d_64", "steps", "noh", [64, 64, 64], 10),
        # a ragged periodic box, eight-point scheme
        _grid("turbulence_3d_ragged", "steps", "turbulence", [150, 97, 133], 8),
        # the 3D turbulence box at its full size
        _grid("turbulence_3d_256", "steps", "turbulence", [256, 256, 256], 10),
        # ensembles of independent shock tubes of uneven length
        _batch("batch_1d_200", 200, 64, 512, 4),
        _batch("batch_1d_4096", 4096, 64, 4096, 1),
        # gradient of a 2D oblique-shock run (checkpointed)
        _grid("rollout_2d_512", "rollout", "oblique", [512, 512], 8, steps=6, every=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs1", "tube", "quadrants", "walls", "turbulence", "turbulence", "noh",
                       "batch", "rollout"])
    scheme = rng.choice([8, 10, 10, 12])
    if kind == "rhs1":
        return _grid(None, "rhs", "tube", [_log(rng, 100, 100000)], scheme,
                     record=rng.random() < 0.3)
    if kind == "tube":
        return _grid(None, "steps", "tube", [_log(rng, 100, 100000)], scheme,
                     steps=rng.randint(1, 10))
    if kind == "quadrants":
        return _grid(None, "steps", "quadrants", [_log(rng, 40, 1200), _log(rng, 40, 1200)], scheme,
                     steps=rng.randint(1, 3))
    if kind == "walls":
        return _grid(None, "rhs", "walls", [_log(rng, 30, 800), _log(rng, 30, 800)], scheme,
                     record=rng.random() < 0.5)
    if kind == "turbulence":
        return _grid(None, "steps", "turbulence", [_log(rng, 20, 200) for _ in range(3)], scheme)
    if kind == "noh":
        n = _log(rng, 28, 96)
        return _grid(None, "steps", "noh", [n, n, n], scheme)
    if kind == "batch":
        lo = _log(rng, 16, 256)
        return _batch(None, _log(rng, 16, 4096), lo, lo * rng.randint(2, 12), rng.randint(1, 3))
    nx, ny = _log(rng, 40, 511), _log(rng, 40, 511)
    # nx + ny even: a stage's decision record, 11 (2 nx ny + nx + ny) bytes,
    # holds 16-bit words, and a step's three records lie back to back
    return _grid(None, "rollout", "oblique", [nx, ny + (nx + ny) % 2], rng.choice([8, 10]),
                 steps=rng.randint(2, 5), every=2)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Random:
    """Seeded numbers: scalars from a CPU generator, fields on the GPU."""

    def __init__(self, seed):
        self.cpu = torch.Generator().manual_seed(int(seed))
        self.gpu = torch.Generator(device=DEV).manual_seed(int(seed))

    def uniform(self, lo, hi):
        return lo + (hi - lo) * torch.rand(1, generator=self.cpu, dtype=F64).item()

    def field(self, shape):
        return torch.rand(shape, generator=self.gpu, dtype=F64, device=DEV)

    def noise(self, x):
        """x with the rounding differences that plateaus carry after some steps."""
        k = torch.randint(-2, 3, x.shape, generator=self.gpu, device=DEV)
        return x * (1.0 + k.to(F64) * 2.0 ** -52)


def _axis(n, length=1.0):
    return (torch.arange(n, dtype=F64, device=DEV) + 0.5) * (length / n)


def _conserved(rho, vel, p, gamma):
    ke = 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (gamma - 1.0) + ke]).contiguous()


def _side(x, x0, width):
    return 0.5 * (1.0 + torch.tanh((x - x0) / width))


def _waves(shape, r, modes=4):
    """A smooth field of a few low Fourier modes, at most 1 in size; shape (nz, ny, nx)."""
    grids = torch.meshgrid(*[_axis(s) for s in shape], indexing="ij")
    out = torch.zeros(shape, dtype=F64, device=DEV)
    for _ in range(modes):
        arg = r.uniform(0, 6.28)
        for g in grids:
            arg = arg + 2 * math.pi * math.floor(r.uniform(1, 4)) * g
        out = out + r.uniform(-1, 1) * torch.sin(arg)
    return out / out.abs().max().clamp_min(1e-3)


def _tube(c, r):
    x = _axis(c["nx"])
    s = _side(x, 0.5, 1.5 / c["nx"])
    q = [(r.uniform(lo, hi), r.uniform(lo, hi)) for lo, hi in ((0.1, 1), (-0.5, 0.5), (0.1, 1))]
    rho, u, p = [a + (b - a) * s for a, b in q]
    rho = rho * (1 + 0.05 * torch.exp(-((x - 0.3) / 0.05) ** 2))
    U = _conserved(r.noise(rho), [u], r.noise(p), 1.4)
    return U, dict(dx=[1.0 / c["nx"]], bc_lo=[TRANSMISSIVE], bc_hi=[TRANSMISSIVE])


def _quadrants(c, r):
    nx, ny = c["nx"], c["ny"]
    sx, sy = _side(_axis(nx), 0.5, 1.5 / nx)[None, :], _side(_axis(ny), 0.5, 1.5 / ny)[:, None]
    f = []
    for lo, hi in ((0.1, 1.5), (-1, 1), (-1, 1), (0.03, 1.5)):
        a, b, d, e = (r.uniform(lo, hi) for _ in range(4))
        f.append((a * (1 - sx) + b * sx) * (1 - sy) + (d * (1 - sx) + e * sx) * sy)
    rho = f[0] * (1 + 0.1 * torch.sin(5 * _axis(nx))[None, :] * (1 - sx) * (1 - sy))
    U = _conserved(r.noise(rho), f[1:3], r.noise(f[3]), 1.4)
    return U, dict(dx=[1.0 / nx, 1.0 / ny], bc_lo=[TRANSMISSIVE] * 2, bc_hi=[TRANSMISSIVE] * 2)


def _walls(c, r):
    nx, ny = c["nx"], c["ny"]
    shape = (ny, nx)
    rho = 1 + 0.3 * _waves(shape, r) + 1e-4 * (r.field(shape) - 0.5)
    p = 1 + 0.3 * _waves(shape, r) + 0.4 * _side(_axis(nx), r.uniform(0.3, 0.7), 1.5 / nx)[None, :]
    U = _conserved(rho, [0.4 * _waves(shape, r), 0.4 * _waves(shape, r)], p, 1.4)
    return U, dict(dx=[1.0 / nx, 1.0 / ny], bc_lo=[NOSLIP, SLIP], bc_hi=[TRANSMISSIVE, SLIP])


def _turbulence(c, r):
    """Mach-0.5 Taylor-Green flow plus solenoidal k^-5/3 noise up to k = 16."""
    n = [c["nz"], c["ny"], c["nx"]]
    Z, Y, X = torch.meshgrid(*[_axis(m, 2 * math.pi) for m in n], indexing="ij")
    vel = [torch.sin(X) * torch.cos(Y) * torch.cos(Z), -torch.cos(X) * torch.sin(Y) * torch.cos(Z),
           torch.zeros_like(X)]
    k = [torch.fft.fftfreq(m, 1.0 / m, dtype=F64, device=DEV) for m in n[:2]]
    k.append(torch.fft.rfftfreq(n[2], 1.0 / n[2], dtype=F64, device=DEV))
    KZ, KY, KX = torch.meshgrid(*k, indexing="ij")
    K2 = KX * KX + KY * KY + KZ * KZ
    amp = torch.where((K2 >= 1) & (K2 <= 256), K2.clamp_min(1.0) ** (-11.0 / 12.0), 0.0)
    h = [amp * r.field(K2.shape) * torch.exp(2j * math.pi * r.field(K2.shape)) for _ in range(3)]
    div = (KX * h[0] + KY * h[1] + KZ * h[2]) / K2.clamp_min(1.0)
    h = [h[0] - KX * div, h[1] - KY * div, h[2] - KZ * div]
    w = [torch.fft.irfftn(a, s=n) for a in h]
    rms = sum(a.square().mean() for a in w).sqrt()
    vel = [v + (0.05 / rms) * a for v, a in zip(vel, w)]
    rho = 1 + 0.02 * torch.sin(X) * torch.sin(Y + 1) * torch.cos(Z)
    U = _conserved(rho, vel, torch.full_like(X, 4.0 / 1.4) * rho ** 1.4, 1.4)
    return U, dict(dx=[2 * math.pi / m for m in reversed(n)], bc_lo=[PERIODIC] * 3,
                   bc_hi=[PERIODIC] * 3)


def _noh(c, r):
    """The 3D Noh implosion at t = 0.3, shock at r = 0.1, inflow through the far faces."""
    n, g, t, L = c["nx"], 5.0 / 3.0, 0.3, 0.256
    shape = (n, n, n)
    x = _axis(n, L)
    Z, Y, X = torch.meshgrid(x, x, x, indexing="ij")
    R = torch.sqrt(X * X + Y * Y + Z * Z)
    s = _side(R, t / 3, L / n)
    ahead = (1 + t / R) ** 2
    rho = (64 * (1 - s) + ahead * s) * (1 + 1e-3 * (r.field(shape) - 0.5))
    p = 64.0 / 3.0 * (1 - s) + 1e-6 * s
    U = _conserved(rho, [-X / R * s, -Y / R * s, -Z / R * s], p, g)
    states = []
    for d in range(3):
        B, A = torch.meshgrid(x, x, indexing="ij")      # (slow, fast) of the other two axes
        q = [A, B]
        q.insert(d, torch.full_like(A, L))
        q = q[:3]
        Rb = torch.sqrt(q[0] ** 2 + q[1] ** 2 + q[2] ** 2)
        ab = (1 + t / Rb) ** 2
        states.append(torch.stack([ab] + [-v / Rb for v in q] + [torch.full_like(Rb, 1e-6)]).reshape(5, -1))
    return U, dict(dx=[L / n] * 3, bc_lo=[SLIP] * 3, bc_hi=[DIRICHLET] * 3, bc_state_hi=states,
                   gamma=g, flux_split=1, limiter=1)


def _oblique(c, r):
    """Mach-2 stationary shock with a tangential velocity, entropy wave and vortex upstream."""
    nx, ny, g = c["nx"], c["ny"], 1.4
    X, Y = _axis(nx)[None, :], _axis(ny)[:, None]
    r2 = (g + 1) * 4 / ((g - 1) * 4 + 2)
    p2 = (1 + 2 * g / (g + 1) * 3) / g
    s = _side(X, 0.5, 1.0 / nx)
    win = 1 - _side(X, 0.38, 0.02)
    rho = 1 + (r2 - 1) * s
    rho = rho * (1 + 0.05 * win * torch.sin(2 * math.pi * (r.uniform(2, 6) * X + 2 * Y)))
    x0, y0 = r.uniform(0.15, 0.3), r.uniform(0.3, 0.7)
    e = 0.95 * win * torch.exp(0.5 - 200 * ((X - x0) ** 2 + (Y - y0) ** 2))
    u = 2 + (2 / r2 - 2) * s - (Y - y0) * e + 1e-3 * _waves((ny, nx), r)
    v = 1 + (X - x0) * e + 1e-3 * _waves((ny, nx), r)
    p = (1 / g + (p2 - 1 / g) * s) * (1 + 1e-3 * _waves((ny, nx), r))
    U = _conserved(rho * (1 + 1e-3 * _waves((ny, nx), r)), [u, v], p, g)
    return U, dict(dx=[1.0 / nx, 1.0 / ny], bc_lo=[TRANSMISSIVE, PERIODIC],
                   bc_hi=[TRANSMISSIVE, PERIODIC])


FIELDS = dict(tube=_tube, quadrants=_quadrants, walls=_walls, turbulence=_turbulence, noh=_noh,
              oblique=_oblique)


def _grid_inputs(c, seed):
    U, o = FIELDS[c["field"]](c, _Random(seed))
    n = [c["nx"], c["ny"], c["nz"]]
    o.update(ndim=U.shape[0] - 2, n=n, scheme=c["scheme"])
    return U.reshape(U.shape[0], -1).contiguous(), o


def _batch_inputs(c, seed):
    """The ensemble's sizes and options, and its packed states of one seed
    (blocks [3][n], 16-byte aligned)."""
    r = _Random(seed)
    count = c["count"]
    plan = torch.Generator().manual_seed(count + 7919 * c["nmax"])
    n = torch.randint(c["nmin"], c["nmax"] + 1, (count,), generator=plan)
    ten, vac = (torch.rand(count, generator=plan) < share for share in (0.5, 0.1))
    u = torch.rand(8, count, generator=r.cpu, dtype=F64)
    rho = 0.1 + 0.9 * u[1:3]
    low = 0.1 + 0.9 * u[3]
    # pressure ratios up to 100, up to 1e5 where the limiter is on
    p = torch.stack([low * torch.exp(u[4] * torch.where(vac, math.log(1e5), math.log(100.0))), low])
    p = torch.where(u[5] < 0.5, p, p.flip(0))
    # near-vacuum side, limiter on
    side = torch.stack([u[7] < 0.5, u[7] >= 0.5]) & vac
    p = torch.where(side, p * (1e-6 / rho), p)
    rho = torch.where(side, torch.full_like(rho, 1e-6), rho)
    start = torch.cat([torch.zeros(1, dtype=torch.int64), ((3 * n + 1) // 2 * 2).cumsum(0)])
    nd = n.to(DEV)
    prob = torch.repeat_interleave(torch.arange(count, device=DEV), nd)
    i = torch.arange(int(n.sum()), device=DEV) - (nd.cumsum(0) - nd)[prob]
    nf = nd[prob].to(F64)
    s = _side((i.to(F64) + 0.5) / nf, 0.5, 1.0 / nf)
    rho, p = rho.to(DEV)[:, prob], p.to(DEV)[:, prob]
    # geometric blends: density and pressure differ by orders of magnitude
    rho = rho[0] * (rho[1] / rho[0]) ** s
    p = p[0] * (p[1] / p[0]) ** s
    U = _conserved(r.noise(rho), [torch.zeros_like(rho)], r.noise(p), 1.4)
    flat = torch.zeros(int(start[-1]), dtype=F64, device=DEV)
    at = start.to(DEV)[prob] + i
    for k in range(3):
        flat[at + k * nd[prob]] = U[k]
    return dict(n=n, start=start, ten=ten, vac=vac, flat=flat, at=at, prob=prob, nd=nd, U=U)


def _max_speeds(U, ndim, gamma):
    rho, E = U[0], U[ndim + 1]
    vel = [U[1 + d] / rho for d in range(ndim)]
    p = (gamma - 1) * (E - 0.5 * sum(U[1 + d] * vel[d] for d in range(ndim)))
    a = torch.sqrt(gamma * p / rho)
    return [v.abs() + a for v in vel]


def prepare(case, seed):
    if case["kind"] == "batch":
        b = _batch_inputs(case, seed)
        problems = [dict(n=n, offset=o, dx=1.0 / n, scheme=10 if t else 8, limiter=int(v),
                         bc_lo=TRANSMISSIVE, bc_hi=TRANSMISSIVE)
                    for n, o, t, v in zip(b["n"].tolist(), b["start"].tolist(), b["ten"].tolist(),
                                          b["vac"].tolist())]
        plan = T.Batch(T.teno_params_init(), problems)
        U = b["flat"].clone()
        plan.autotune(U)
        return dict(case=case, plan=plan, U0=b["flat"], U=U)
    U0, o = _grid_inputs(case, seed)
    s = dict(case=case, U0=U0, U=torch.empty_like(U0), keep=o.get("bc_state_hi"))
    p = s["p"] = T.teno_params_init(**o)
    if case["kind"] == "rollout":
        A = _max_speeds(U0, p.ndim, p.gamma)
        s["dt"] = 0.4 / sum(a.max().item() / dx for a, dx in zip(A, o["dx"]))
        s["target"] = U0[0] * (1 + 1e-3 * _waves((case["ny"], case["nx"]), _Random(seed + 1)).reshape(-1))
    else:
        s["solver"] = T.Solver(p)
    return s


def run(state):
    case, U0, U = state["case"], state["U0"], state["U"]
    if case["kind"] == "rhs":
        # the limiter is off in these cases, so its time step is not used
        out = state["solver"].rhs(U0, flags=case["record"])
        return list(out) if case["record"] else out
    if case["kind"] == "rollout":
        x = U0.detach().requires_grad_(True)
        end = T.rollout(state["p"], x, state["dt"], case["steps"], case["every"])
        loss = (end[0] - state["target"]).square().mean()
        grad, = torch.autograd.grad(loss, x)
        return [end.detach(), grad]
    U.copy_(U0)
    if case["kind"] == "batch":
        state["plan"].steps(U, case["steps"], 0.4)
        return U
    for _ in range(case["steps"]):
        dt = state["solver"].cfl_dt(U, 0.4)
        state["solver"].step(U)
    return [U, dt]


def work(case):
    """One pass at FP64: per face, field and sign the projection, the split and
    one linear scheme, and the Roe state; per cell the state in and out, and
    what the record or the adjoint adds."""
    if case["kind"] == "batch":
        cells, nd, W = case["count"] * (case["nmin"] + case["nmax"]) / 2, 1, 9
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        nd, W = 1 + (case["ny"] > 1) + (case["nz"] > 1), case["scheme"]
    nc = nd + 2
    face = 60 + W * nc * (4 * nc + 4) + 2 * nc * (2 * W - 1)
    stages = 1 if case["kind"] == "rhs" else 3 * case["steps"]
    flops = cells * nd * face * stages
    byts = 16.0 * nc * cells
    if case["kind"] == "rhs" and case["record"]:
        byts += cells * nd * (2 * nc + 3)
    if case["kind"] == "rollout":
        flops *= 3
        byts += 16.0 * cells + 8.0 * nc * cells
    return dict(bytes=byts, flops=flops)


# ---------------------------------------------------------------------------
# the same outputs from the formulas, plain FP64 PyTorch
# ---------------------------------------------------------------------------

LINEAR = {
    3: [0.02852274270130377, -0.1714015614372447, 0.650378818735941, 0.6253788187359414,
        -0.1589015614372448, 0.02602274270130375],
    4: [-0.006866688980568011, 0.05128582585522106, -0.1968478198727312, 0.6552858258552222,
        0.6452858258552218, -0.1908478198727314, 0.04928582585522098, -0.006580974694853729],
    5: [0.001911786299492748, -0.0170332977472532, 0.07339445614860979, -0.221228429084247,
        0.6657332621611695, 0.6557332621611695, -0.2145617624175796, 0.07053731329146805,
        -0.01631901203296621, 0.001832421220128962],
    6: [float.fromhex(h) for h in (
        "-0x1.18c591608ba4ep-11", "0x1.714ca8699bc8dp-8", "-0x1.cc2d4b3d96aacp-6",
        "0x1.76ee011841e20p-4", "-0x1.e86f451607ff3p-3", "0x1.58688ba642e5ap-1",
        "0x1.5349d35457608p-1", "-0x1.d9ce5b0767153p-3", "0x1.684d1709a0f7fp-4",
        "-0x1.b8ac132a1572bp-6", "0x1.61b21526ce026p-8", "-0x1.0d6c6c18b02bdp-11")],
}
SMALL = [[0, -1 / 6, 5 / 6, 2 / 6, 0], [0, 0, 2 / 6, 5 / 6, -1 / 6], [2 / 6, -7 / 6, 11 / 6, 0, 0]]
WEIGHTS = [0.5065006634, 0.3699651429, 0.1235341937]
CHUNK = 1 << 21                       # faces evaluated at a time


@functools.lru_cache(None)
def _indicator(L):
    """Smoothness indicator of offsets 1-L..L: sum over l >= 1 of the integral
    over cell 0 of (d^l p / dx^l)^2, p with those cell averages, as a matrix."""
    offs = range(1 - L, L + 1)
    n = 2 * L
    rows = [[(Fraction(2 * o + 1, 2) ** (k + 1) - Fraction(2 * o - 1, 2) ** (k + 1)) / (k + 1)
             for k in range(n)] + [Fraction(int(i == j)) for j in range(n)]
            for i, o in enumerate(offs)]
    for c in range(n):                                # Gauss-Jordan
        piv = next(r for r in range(c, n) if rows[r][c])
        rows[c], rows[piv] = rows[piv], rows[c]
        rows[c] = [v / rows[c][c] for v in rows[c]]
        for r in range(n):
            if r != c and rows[r][c]:
                f = rows[r][c]
                rows[r] = [a - f * b for a, b in zip(rows[r], rows[c])]
    coef = [row[n:] for row in rows]                  # coef[k][j]: x^k from average j
    B = [[Fraction(0)] * n for _ in range(n)]
    for l in range(1, n):
        fall = [math.prod(range(k - l + 1, k + 1)) for k in range(n)]
        for a in range(l, n):
            for b in range(l, n):
                e = a + b - 2 * l
                if e % 2:
                    continue
                w = fall[a] * fall[b] * Fraction(2, (e + 1) * 2 ** (e + 1))
                for i in range(n):
                    t = w * coef[a][i]
                    for j in range(n):
                        B[i][j] += t * coef[b][j]
    return [[float(v) for v in row] for row in B]


@functools.lru_cache(None)
def _schemes(H):
    """Rows of linear coefficients on offsets 1-H..H: 0-7 the fallback blends by
    their cut-off bits, 8 + L the large stencils."""
    rows = torch.zeros(8 + H + 1, 2 * H, dtype=F64)
    for mask in range(1, 8):
        w = [d if mask >> k & 1 else 0.0 for k, d in enumerate(WEIGHTS)]
        for k in range(3):
            rows[mask, H - 3:H + 2] += w[k] / sum(w) * torch.tensor(SMALL[k], dtype=F64)
    for L in range(3, H + 1):
        rows[8 + L, H - L:H + L] = torch.tensor(LINEAR[L], dtype=F64)
    return rows.to(DEV)


def _decide(v, H):
    """Row of _schemes(H) that TENO-AA selects for the values v[offset + H - 1]."""
    V = lambda m: v[m + H - 1]  # noqa: E731
    eps = 1e-40
    dl = [V(m + 1) - V(m) for m in range(-2, 3)]
    eta = None
    for j in range(1, 5):
        e = ((2 * dl[j] * dl[j - 1]).abs() + eps) / (dl[j] ** 2 + dl[j - 1] ** 2 + eps)
        eta = e if eta is None else torch.minimum(eta, e)
    m = 1 - (eta / 0.265).clamp_max(1.0)
    g = (1 - m) ** 4 * (1 + 4 * m)
    # the values across two problems of a batch, which nothing uses, may be no numbers
    n = torch.floor(14.0 - 6.4 * (1 - g)).clamp(0, 22).nan_to_num(0.0).long()
    CT = torch.tensor([float("1e-%d" % k) for k in range(23)], dtype=F64, device=DEV)[n]
    pairs = [(V(-1) - V(1), V(-1) - 2 * V(0) + V(1)),
             (3 * V(0) - 4 * V(1) + V(2), V(0) - 2 * V(1) + V(2)),
             (V(-2) - 4 * V(-1) + 3 * V(0), V(-2) - 2 * V(-1) + V(0))]
    gam = [1 / (0.25 * a * a + 13.0 / 12.0 * b * b + eps) ** 7 for a, b in pairs]
    s = gam[0] + gam[1] + gam[2]
    code = sum(((x / s) >= CT).long() << k for k, x in enumerate(gam))
    for L in range(3, H + 1):                         # the largest accepted one wins
        B = _indicator(L)
        sh = {o: V(o) - V(0) for o in range(1 - L, L + 1) if o}
        beta = 0
        for i in sh:
            beta = beta + sh[i] * sum(B[i + L - 1][j + L - 1] * sh[j] for j in sh)
        x = 1 / (beta + eps) ** 7
        code = torch.where((x / (s + x)) >= CT, 8 + L, code)
    return code


def _recon(v, H):
    with torch.no_grad():
        c = _schemes(H)[_decide(v, H)]
    return sum(c[..., k] * v[k] for k in range(2 * H))


def _cell(U, d, gamma):
    nd = U.shape[0] - 2
    vel = [U[1 + a] / U[0] for a in range(nd)]
    p = (gamma - 1) * (U[-1] - 0.5 * sum(U[1 + a] * vel[a] for a in range(nd)))
    F = [U[1 + d]] + [U[1 + d] * vel[a] + (p if a == d else 0) for a in range(nd)]
    return vel, p, torch.sqrt(gamma * p / U[0]), (U[-1] + p) / U[0], F + [vel[d] * (U[-1] + p)]


def _faces(P, d, H, o, lam=None, limited=None):
    """Face fluxes from cells with ghosts P [nc, cells + 2H, pencils]: faces + 1."""
    gamma, nd = o.get("gamma", 1.4), P.shape[0] - 2
    nc, W, nf = nd + 2, 2 * H, P.shape[1] - 2 * H + 1
    at = lambda q, j: q[j:j + nf]  # noqa: E731
    vel, p, a, Ht, F = _cell(P, d, gamma)
    sr = torch.sqrt(P[0])
    sl, s_r = at(sr, H - 1), at(sr, H)
    roe = lambda q: (sl * at(q, H - 1) + s_r * at(q, H)) / (sl + s_r)  # noqa: E731
    u, h = [roe(v) for v in vel], roe(Ht)
    q2 = sum(x * x for x in u)
    c = torch.sqrt((gamma - 1) * (h - 0.5 * q2))
    un, b1 = u[d], (gamma - 1) / (c * c)
    b2 = 0.5 * q2 * b1
    tang = [x for x in range(nd) if x != d]
    one, zero = torch.ones_like(un), torch.zeros_like(un)

    def acoustic(sg):                                 # u + sg c
        l = [0.5 * (b2 - sg * un / c)] + [0.5 * ((sg / c if x == d else 0) - b1 * u[x])
                                          for x in range(nd)] + [0.5 * b1]
        r = [one] + [u[x] + (sg * c if x == d else 0) for x in range(nd)] + [h + sg * un * c]
        return l, r

    fields = [acoustic(-1.0),
              ([1 - b2] + [b1 * x for x in u] + [-b1], [one] + u + [0.5 * q2])]
    for t in tang:
        e = [one if x == t else zero for x in range(nd)]
        fields.append(([-u[t]] + e + [zero], [zero] + e + [u[t]]))
    fields.append(acoustic(1.0))
    # a ghost cell whose pressure is below zero has no speed and does not count
    wide = lambda q: torch.stack([at(q, j) for j in range(W)]).nan_to_num(0.0).amax(0)  # noqa: E731
    if o.get("flux_split", 0):
        alphas = [wide(vel[d].abs() + a)] * nc
    else:
        mid = wide(vel[d].abs())
        alphas = [wide((vel[d] - a).abs())] + [mid] * nd + [wide((vel[d] + a).abs())]
    out = [0] * nc
    for (l, r), al in zip(fields, alphas):
        w = [sum(l[k] * at(P[k], j) for k in range(nc)) for j in range(W)]
        g = [sum(l[k] * at(F[k], j) for k in range(nc)) for j in range(W)]
        hh = _recon([0.5 * (y + al * x) for x, y in zip(w, g)], H) + \
            _recon([0.5 * (y - al * x) for x, y in zip(w, g)][::-1], H)
        out = [q + r[k] * hh for k, q in enumerate(out)]
    out = torch.stack(out)
    if lam is None:
        return out
    # positivity limiter: blend toward the Lax-Friedrichs flux (eps = 1e-13)
    eps, F = 1e-13, torch.stack(F)
    Ul, Ur, Fl, Fr = P[:, H - 1:H - 1 + nf], P[:, H:H + nf], F[:, H - 1:H - 1 + nf], F[:, H:H + nf]
    sp = (vel[d].abs() + a).nan_to_num(0.0)
    LF = 0.5 * (Fl + Fr - torch.maximum(at(sp, H - 1), at(sp, H)) * (Ur - Ul))
    pres = lambda q: (gamma - 1) * (q[-1] - 0.5 * (q[1:-1] ** 2).sum(0) / q[0])  # noqa: E731
    states = [(Ul - 2 * lam * (LF - Fl), -2 * lam * (out - LF)),
              (Ur + 2 * lam * (LF - Fr), 2 * lam * (out - LF))]
    th = one
    for q, dq in states:
        t = (q[0] - eps) / -dq[0]
        t = torch.where(t > 0, t, 0.0)
        th = torch.where(q[0] + dq[0] < eps, torch.minimum(th, t), th)
    thp = th
    for q, dq in states:
        pt, p0 = pres(q + th * dq), pres(q)
        t = th * ((p0 - eps) / (p0 - pt))
        t = torch.where(t > 0, t, 0.0)
        thp = torch.where(pt < eps, torch.minimum(thp, t), thp)
    if limited is not None:
        thp = torch.where(limited, thp, one)
    return torch.where(thp < 1, LF + thp * (out - LF), out)


def _ghosts(V, d, H, o):
    """V [nc, cells along d, pencils] with H ghost cells at both ends (App. A)."""
    gamma, nd, n = o.get("gamma", 1.4), V.shape[0] - 2, V.shape[1]
    ends = []
    for side in (0, 1):
        rule = o["bc_hi" if side else "bc_lo"][d]
        if rule == PERIODIC:
            ends.append(V[:, :H] if side else V[:, n - H:])
            continue
        if rule == TRANSMISSIVE:
            ends.append(V[:, -1:].expand(-1, H, -1) if side else V[:, :1].expand(-1, H, -1))
            continue
        M = V[:, n - H:].flip(1) if side else V[:, :H].flip(1)
        if rule == DIRICHLET:
            b = o["bc_state_hi" if side else "bc_state_lo"][d][:, None, :]
            vel = [2 * b[1 + a] - M[1 + a] / M[0] for a in range(nd)]
            p = 2 * b[-1] - (gamma - 1) * (M[-1] - 0.5 * (M[1:-1] ** 2).sum(0) / M[0])
            ends.append(_conserved(2 * b[0] - M[0], vel, p, gamma))
            continue
        s = torch.ones(V.shape[0], 1, 1, dtype=F64, device=DEV)
        if rule == NOSLIP:
            s[1:-1] = -1
        else:
            s[1 + d] = -1
        ends.append(M * s)
    return torch.cat([ends[0], V, ends[1]], 1)


def _rhs(U, o, dt=None):
    """L(U) of a grid state [nc, cells]."""
    n, nd, H, out = o["n"], o["ndim"], o["scheme"] // 2, 0
    grid = U.reshape(nd + 2, n[2], n[1], n[0])
    lam = [None] * nd
    if o.get("limiter"):
        A = [s.max() for s in _max_speeds(U, nd, o.get("gamma", 1.4))]
        S = sum(x / dx for x, dx in zip(A, o["dx"]))
        lam = [dt / o["dx"][0]] if nd == 1 else [dt * S / x for x in A]
    for d in range(nd):
        V = grid.movedim(3 - d, 1)
        V = V.reshape(nd + 2, n[d], -1)               # other axes keep their order, x fastest
        P = _ghosts(V, d, H, o)
        step = max(1, CHUNK // n[d])
        F = torch.cat([_faces(P[:, :, k:k + step], d, H, o, lam[d])
                       for k in range(0, P.shape[2], step)], 2)
        R = (F[:, 1:] - F[:, :-1]) / -o["dx"][d]
        shape = [n[a] for a in (2, 1, 0) if a != d]
        out = out + R.reshape([nd + 2, n[d]] + shape).movedim(1, 3 - d)
    return out.reshape(nd + 2, -1)


def _batch_rhs(U, b, dt):
    """L(U) of every problem of a batch, U [3, all cells]; transmissive ends."""
    out = torch.empty_like(U)
    for ten, H in ((False, 4), (True, 5)):
        mine = (b["ten"] == ten).nonzero().flatten().to(DEV)
        if not len(mine):
            continue
        n = b["nd"][mine]
        first = (b["nd"].cumsum(0) - b["nd"])[mine]
        which = torch.repeat_interleave(torch.arange(len(mine), device=DEV), n + 2 * H)
        ends = (n + 2 * H).cumsum(0)
        j = torch.arange(int(ends[-1]), device=DEV) - (ends - n - 2 * H)[which] - H
        P = U[:, first[which] + torch.minimum(j.clamp_min(0), n[which] - 1)]
        face = which[H:len(which) - H + 1]            # face f: right face of the padded cell f + H - 1
        lam = (dt * b["nd"])[mine][face]              # dt / dx
        F = _faces(P[:, :, None], 0, H, {}, lam[:, None], b["vac"].to(DEV)[mine][face][:, None])
        cell = ((j >= 0) & (j < n[which])).nonzero().flatten()
        R = -(F[:, cell - H + 1, 0] - F[:, cell - H, 0]) * n[which[cell]]
        out[:, first[which[cell]] + j[cell]] = R
    return out


def _rk3(U, dt, L):
    U1 = U + dt * L(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * L(U1))
    return U / 3 + (U2 + dt * L(U2)) * (2.0 / 3.0)


def exact(case, seed):
    if case["kind"] == "batch":
        b = _batch_inputs(case, seed)
        U = b["U"]
        for _ in range(case["steps"]):
            A = torch.zeros(case["count"], dtype=F64, device=DEV)
            A.scatter_reduce_(0, b["prob"], _max_speeds(U, 1, 1.4)[0], "amax")
            dt = 0.4 / (A * b["nd"])
            U = _rk3(U, dt[b["prob"]], lambda V: _batch_rhs(V, b, dt))
        flat = torch.zeros_like(b["flat"])
        for k in range(3):
            flat[b["at"] + k * b["nd"][b["prob"]]] = U[k]
        return flat
    U, o = _grid_inputs(case, seed)
    if case["kind"] == "rhs":
        r = _rhs(U, o)
        return [r, None] if case["record"] else r
    if case["kind"] == "rollout":
        A = _max_speeds(U, o["ndim"], 1.4)
        dt = 0.4 / sum(a.max().item() / dx for a, dx in zip(A, o["dx"]))
        target = U[0] * (1 + 1e-3 * _waves((case["ny"], case["nx"]), _Random(seed + 1)).reshape(-1))
        x = U.detach().requires_grad_(True)
        end = x
        for _ in range(case["steps"]):
            end = torch.utils.checkpoint.checkpoint(
                lambda V: _rk3(V, dt, lambda q: _rhs(q, o)), end, use_reentrant=False)
        grad, = torch.autograd.grad((end[0] - target).square().mean(), x)
        return [end.detach(), grad]
    for _ in range(case["steps"]):
        A = _max_speeds(U, o["ndim"], o.get("gamma", 1.4))
        dt = 0.4 / sum(a.max() / dx for a, dx in zip(A, o["dx"]))
        U = _rk3(U, dt, lambda q: _rhs(q, o, dt))
    return [U, dt.reshape(1)]
