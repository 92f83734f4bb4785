"""Routes that small grids do not reach, against the oracle, bitwise: the four
face-flux kernels with walls, Dirichlet sides, the limiter and larger epsilons
in 1D and 2D; the single launch in 3D; the right-hand side without a workspace
in several pieces; a batch above the fused stages' limit in every mode.  Each
case checks the tile count that puts it on its route."""
import numpy as np
import pytest

import oracle
import workloads
from helpers import oracle_params, tiles_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T  # noqa: E402


def one_launch_most(case):
    return {1: 4096, 2: 1024 if case["scheme"] == 12 else 3072, 3: 512}[case["ndim"]]


def gpu_params(case, **kw):
    keep = []
    for side in ("bc_state_lo", "bc_state_hi"):
        if case.get(side) is not None:
            kw[side] = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
                        for a in case[side]]
            keep += kw[side]
    p = T.teno_params_init(ndim=case["ndim"], n=case["n"], dx=case["dx"], scheme=case["scheme"],
                           gamma=case["gamma"], bc_lo=case["bc_lo"], bc_hi=case["bc_hi"],
                           limiter=case.get("limiter", 0), **kw)
    p._keep = keep
    return p


def compare(case, eps=None, step=True):
    kw = {} if eps is None else dict(eps_beta=eps, eps_eta=eps)
    p, po = gpu_params(case, **kw), oracle_params(case, **kw)
    s = T.Solver(p)
    U = torch.from_numpy(np.ascontiguousarray(case["U"])).cuda()
    dt, _, _ = oracle.cfl_dt(po, case["U"], 0.4)
    r_o, f_o, l_o, _ = oracle.rhs(po, case["U"], dt, want_flags=True, threads=8)
    plain = s.rhs(U, dt)
    rec, fl = s.rhs(U, dt, flags=True)
    assert np.array_equal(plain.cpu().numpy(), r_o)
    assert torch.equal(rec, plain)
    assert np.array_equal(fl.cpu().numpy()[:f_o.size], f_o)
    if step:
        U1, _ = oracle.rk3_step(po, case["U"], dt, threads=8)
        s.step(U, dt)
        assert np.array_equal(U.cpu().numpy(), U1)
    s.status()


FOUR = {
    "1d-noslip-dirichlet-s8": lambda: workloads.boundary_walls(1, [131500], [3], [4], scheme=8),
    "1d-slip-s12": lambda: workloads.boundary_walls(1, [131200], [2], [1], scheme=12),
    "1d-limiter-s10": lambda: dict(workloads.double_rarefaction_1d(131300, scheme=10), limiter=1),
    "2d-noslip-dirichlet-s10": lambda: workloads.boundary_walls(2, [233, 227], [3, 4], [4, 2], scheme=10),
    "2d-slip-s12": lambda: workloads.boundary_walls(2, [141, 131], [2, 3], [2, 1], scheme=12),
    "2d-limiter-s8": lambda: dict(workloads.quadrants_2d(239, 231, scheme=8), limiter=1),
}


@pytest.mark.parametrize("name", FOUR)
def test_four_kernels(name):
    case = FOUR[name]()
    assert tiles_of(case) > one_launch_most(case)
    compare(case)


EPS = {
    "1d-s8": lambda: workloads.riemann_1d(131100, scheme=8),
    "1d-smooth-s10": lambda: workloads.smooth_wave_1d(131100, 10, amp=1e-3),
    "2d-s10": lambda: workloads.quadrants_2d(229, 231, scheme=10),
    "2d-s12": lambda: workloads.adjoint_2d(139, 133, scheme=12),
    "3d-s8": lambda: workloads.tgv_3d(22, scheme=8),
}


@pytest.mark.parametrize("eps", [1e-6, 1e-20])
@pytest.mark.parametrize("name", EPS)
def test_four_kernels_epsilons(name, eps):
    case = EPS[name]()
    assert tiles_of(case) > one_launch_most(case)
    compare(case, eps=eps, step=False)


@pytest.mark.parametrize("scheme", [8, 10, 12])
def test_one_launch_3d(scheme):
    case = workloads.boundary_walls(3, [16, 15, 14], [2, 3, 0], [1, 2, 0], scheme=scheme)
    assert tiles_of(case) <= one_launch_most(case)
    compare(case)


PIECES = {
    "1d": lambda: workloads.smooth_wave_1d(500000, 10, amp=1e-3),
    "2d": lambda: workloads.quadrants_2d(400, 400, scheme=10),
    "3d": lambda: workloads.tgv_3d(48, scheme=10),
}


@pytest.mark.parametrize("name", PIECES)
def test_static_pieces(name):
    """192 MiB hold, per tile of 32 faces, room for 64 nc queued reconstructions
    (2H values, slot, list entry) beside the faces' values and Roe states."""
    case = PIECES[name]()
    nd, nc, W = case["ndim"], case["ndim"] + 2, case["scheme"]
    tile = 64 * nc * (8 * W + 4 + 2) + 4 + 32 * (8 * 2 * nc + 8 * (nd + 4) + 2 * nc)
    assert tiles_of(case) > (192 << 20) // tile
    p = gpu_params(case)
    U = torch.from_numpy(np.ascontiguousarray(case["U"])).cuda()
    r_o, f_o, _, _ = oracle.rhs(oracle_params(case), case["U"], want_flags=True, threads=8)
    out, rec = torch.empty_like(U), torch.empty_like(U)
    fl = torch.zeros(T.teno_flags_bytes(p), dtype=torch.uint8, device="cuda")
    T.teno_rhs_static(p, U, out, 0.0, None)
    T.teno_rhs_static(p, U, rec, 0.0, fl)
    assert np.array_equal(out.cpu().numpy(), r_o)
    assert torch.equal(rec, out)
    assert np.array_equal(fl.cpu().numpy()[:f_o.size], f_o)


def make_batch():
    """300 problems of 64 to 512 cells: more tiles than the fused stages take (2400)."""
    cases = workloads.batched_1d(count=300, nmin=64, nmax=512)
    assert sum(-(-c["n"][0] // 31) for c in cases) > 2400
    offs, total = T.pack_offsets([c["n"][0] for c in cases])
    U, probs = np.zeros(total), []
    for c, o in zip(cases, offs):
        n = c["n"][0]
        U[o:o + 3 * n] = c["U"].ravel()
        probs.append(dict(n=n, offset=o, dx=c["dx"][0], scheme=c["scheme"], limiter=c["limiter"],
                          bc_lo=1, bc_hi=1))
    return cases, offs, probs, U


def test_batch_modes():
    cases, offs, probs, U = make_batch()
    got = {}
    for mode in (T.TENO_BATCH_GRAPH, T.TENO_BATCH_STREAM, T.TENO_BATCH_PER_PROBLEM):
        B = T.Batch(T.teno_params_init(gamma=1.4), probs)
        Ud = torch.from_numpy(U).cuda()
        B.steps(Ud, 2, 0.4, mode)
        got[mode] = Ud.cpu().numpy()
    assert np.array_equal(got[T.TENO_BATCH_GRAPH], got[T.TENO_BATCH_STREAM])
    assert np.array_equal(got[T.TENO_BATCH_GRAPH], got[T.TENO_BATCH_PER_PROBLEM])
    for c, o in zip(cases, offs):
        po, Uo = oracle_params(c), c["U"].copy()
        for _ in range(2):
            Uo, _ = oracle.rk3_step(po, Uo, oracle.cfl_dt(po, Uo, 0.4)[0])
        assert np.array_equal(got[T.TENO_BATCH_GRAPH][o:o + Uo.size].reshape(Uo.shape), Uo)


def test_batch_autotune_and_replay():
    cases, offs, probs, U = make_batch()
    B = T.Batch(T.teno_params_init(gamma=1.4), probs)
    tile, bps = B.autotune(torch.from_numpy(U).cuda())
    assert tile in (64, 128, 256) and bps in (1, 2, 3, 4, 6)
    Ud = torch.from_numpy(U).cuda()
    B.steps(Ud, 1, 0.4, T.TENO_BATCH_GRAPH)
    Ud.copy_(torch.from_numpy(U))                        # same buffer, new contents
    B.steps(Ud, 2, 0.4, T.TENO_BATCH_GRAPH)
    B2 = T.Batch(T.teno_params_init(gamma=1.4), probs)
    Ud2 = torch.from_numpy(U).cuda()
    B2.steps(Ud2, 2, 0.4, T.TENO_BATCH_STREAM)
    assert torch.equal(Ud, Ud2)
