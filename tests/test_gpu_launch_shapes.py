"""Sizes on both sides of where the launches change: an evaluation in one launch
(fused with the stage update in 1D) or over four kernels, a batch's fused stages,
its two schemes' decisions together or apart, and the fixed scratch's pieces.
Every value and decision byte must be the oracle's, bitwise: each route forms the
same expressions in the same order."""
import numpy as np
import pytest

import oracle
import workloads
from helpers import oracle_params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T  # noqa: E402

CASES = {
    "1d-4096-tiles": lambda: workloads.riemann_1d(131071, scheme=8),
    "1d-4097-tiles": lambda: workloads.riemann_1d(131072, scheme=10),
    "2d-one-launch": lambda: workloads.quadrants_2d(217, 211, scheme=10),
    "2d-four-kernels": lambda: workloads.quadrants_2d(241, 229, scheme=8),
    "2d-one-launch-s12": lambda: workloads.adjoint_2d(121, 119, scheme=12),
    "2d-four-kernels-s12": lambda: workloads.adjoint_2d(139, 133, scheme=12),
    "3d-one-launch": lambda: workloads.boundary_walls(3, [17, 16, 15], [2, 3, 0], [1, 2, 0], scheme=8),
    "3d-four-kernels": lambda: workloads.boundary_walls(3, [21, 19, 17], [0, 2, 3], [0, 1, 2], scheme=10),
    "3d-four-kernels-s12": lambda: workloads.boundary_walls(3, [23, 18, 19], [2, 0, 1], [2, 0, 1], scheme=12),
}


@pytest.mark.parametrize("name", CASES)
def test_both_sides_of_the_launch_rule(name):
    case = CASES[name]()
    p = T.teno_params_init(ndim=case["ndim"], n=case["n"], dx=case["dx"], scheme=case["scheme"],
                           gamma=case["gamma"], bc_lo=case["bc_lo"], bc_hi=case["bc_hi"])
    po = oracle_params(case)
    s = T.Solver(p)
    U = torch.from_numpy(np.ascontiguousarray(case["U"])).cuda()
    r_o, f_o, _, _ = oracle.rhs(po, case["U"], want_flags=True, threads=8)
    plain = s.rhs(U, 0.0)
    rec, fl = s.rhs(U, 0.0, flags=True)
    static = torch.empty_like(U)
    T.teno_rhs_static(p, U, static, 0.0, None)
    assert np.array_equal(plain.cpu().numpy(), r_o)
    assert torch.equal(rec, plain) and torch.equal(static, plain)
    assert np.array_equal(fl.cpu().numpy()[:f_o.size], f_o)
    dt, _, _ = oracle.cfl_dt(po, case["U"], 0.4)
    U1, _ = oracle.rk3_step(po, case["U"], dt, threads=8)
    s.step(U, dt)
    assert s.status() == 0
    assert np.array_equal(U.cpu().numpy(), U1)


@pytest.mark.parametrize("count", [180, 300, 420], ids=["fused", "together", "apart"])
def test_batch_routes(count):
    """1689 tiles of 31 cells (the fused stage takes up to 2400), 2833 and 4636 of 32
    faces (both schemes' decisions go together up to 4096)."""
    cases = workloads.batched_1d(count=count, nmin=64, nmax=600 if count == 420 else 512)
    offs, total = T.pack_offsets([c["n"][0] for c in cases])
    U = np.zeros(total)
    probs = []
    for c, o in zip(cases, offs):
        n = c["n"][0]
        U[o:o + 3 * n] = c["U"].ravel()
        probs.append(dict(n=n, offset=o, dx=c["dx"][0], scheme=c["scheme"],
                          limiter=c.get("limiter", 0), bc_lo=c["bc_lo"][0], bc_hi=c["bc_hi"][0]))
    B = T.Batch(T.teno_params_init(gamma=1.4), probs)
    Ud = torch.from_numpy(U).cuda()
    B.steps(Ud, 2, 0.4, T.TENO_BATCH_GRAPH)
    g = Ud.cpu().numpy()
    for c, o in zip(cases, offs):
        po, Uo = oracle_params(c), c["U"].copy()
        for _ in range(2):
            Uo, _ = oracle.rk3_step(po, Uo, oracle.cfl_dt(po, Uo, 0.4)[0])
        n = c["n"][0]
        assert np.array_equal(g[o:o + 3 * n].reshape(3, n), Uo)
