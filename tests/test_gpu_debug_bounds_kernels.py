"""The bounds-checked build on grids and batches large enough for the four
face-flux kernels (test_gpu_debug_bounds.py runs small ones, which take the
single launch): plain and recording sweeps, decide, exact, finish, the
limiter's rows, frozen replays, combine, and a batch's persistent sweep with
its two schemes' decisions together and apart.  No range check may fail, and
the results are the oracle's, bitwise.

The checked library is built and run in a child process (TENO_GB300_DEBUG=1
selects it in the binding; a process loads one build)."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def test_bounds_checked_kernels():
    env = dict(os.environ, TENO_GB300_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=env, capture_output=True,
                       text=True, timeout=1200, cwd=ROOT)
    assert r.returncode == 0, (r.stdout[-3000:], r.stderr[-3000:])
    res = json.loads([l for l in r.stdout.splitlines() if l.startswith("{")][-1])
    assert res == dict(cases=9, out_of_range=[], not_bitwise=[]), res


def _child():
    from paper_2109_14340_gb300 import _build
    _build.build(debug=True)
    import oracle
    import workloads
    from helpers import oracle_params, tiles_of
    import paper_2109_14340_gb300 as T
    assert T.teno_build_flags() == 1
    out = dict(cases=0, out_of_range=[], not_bitwise=[])

    def done(name, ws, same):
        n, line, idx, ext = T.teno_debug_bounds(ws)
        if n:
            out["out_of_range"].append((name, n, line, idx, ext))
        if not same:
            out["not_bitwise"].append(name)
        out["cases"] += 1

    def grid(name, c, above, limiter=0):
        keep = {}
        for side in ("bc_state_lo", "bc_state_hi"):
            if c.get(side) is not None:
                keep[side] = [None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
                              for a in c[side]]
        c["limiter"] = limiter
        p = T.teno_params_init(ndim=c["ndim"], n=c["n"], dx=c["dx"], scheme=c["scheme"], gamma=c["gamma"],
                               bc_lo=c["bc_lo"], bc_hi=c["bc_hi"], limiter=limiter, **keep)
        assert tiles_of(c) > above                       # four kernels
        po = oracle_params(c)
        s = T.Solver(p)
        U = torch.from_numpy(np.ascontiguousarray(c["U"])).cuda()
        dt, _, _ = oracle.cfl_dt(po, c["U"], 0.4)
        r, fl = s.rhs(U, dt, flags=True)
        ro, fo, _, _ = oracle.rhs(po, c["U"], dt, want_flags=True, threads=8)
        same = np.array_equal(r.cpu().numpy(), ro) and np.array_equal(fl.cpu().numpy()[:fo.size], fo)
        rf = torch.empty_like(U)
        T.teno_rhs_frozen(p, U, rf, fl, s.ws, dt)
        scale = r.abs().amax(dim=1, keepdim=True)
        same = same and float(((rf - r).abs() / scale).max()) <= 1e-13     # as the frozen tests have it
        s.step(U, dt)
        same = same and np.array_equal(U.cpu().numpy(), oracle.rk3_step(po, c["U"], dt, threads=8)[0])
        s.status()
        done(name, s.ws, same)

    grid("1d", workloads.riemann_1d(140001, scheme=8), 4096)
    grid("1d-limiter", workloads.double_rarefaction_1d(135000, scheme=10), 4096, limiter=1)
    grid("2d", workloads.quadrants_2d(241, 229, scheme=8), 3072)
    grid("2d-s12", workloads.adjoint_2d(139, 133, scheme=12), 1024)
    grid("2d-dirichlet", workloads.boundary_walls(2, [233, 227], [3, 4], [2, 4], scheme=10), 3072)
    grid("3d-limiter", workloads.boundary_walls(3, [23, 18, 19], [2, 0, 4], [3, 0, 1], scheme=10), 512,
         limiter=1)
    for count, nmax in ((300, 512), (420, 600)):         # decisions together, apart
        cases = workloads.batched_1d(count=count, nmin=64, nmax=nmax)
        offs, total = T.pack_offsets([c["n"][0] for c in cases])
        Uh, probs = np.zeros(total), []
        for c, o in zip(cases, offs):
            n = c["n"][0]
            Uh[o:o + 3 * n] = c["U"].ravel()
            probs.append(dict(n=n, offset=o, dx=c["dx"][0], scheme=c["scheme"], limiter=c["limiter"],
                              bc_lo=1, bc_hi=1))
        B = T.Batch(T.teno_params_init(gamma=1.4), probs)
        Ub = torch.from_numpy(Uh).cuda()
        B.steps(Ub, 1, 0.4, T.TENO_BATCH_STREAM)
        g = Ub.cpu().numpy()
        same = True
        for c, o in zip(cases, offs):
            po = oracle_params(c)
            Uo, _ = oracle.rk3_step(po, c["U"], oracle.cfl_dt(po, c["U"], 0.4)[0])
            same = same and np.array_equal(g[o:o + Uo.size].reshape(Uo.shape), Uo)
        done("batch-%d" % count, B.ws, same)
    # the reverse kernels stage their cells as the sweeps do
    c = workloads.adjoint_2d(64, 48)
    p = T.teno_params_init(ndim=2, n=c["n"], dx=c["dx"], scheme=8, bc_lo=c["bc_lo"], bc_hi=c["bc_hi"])
    U = torch.from_numpy(c["U"]).cuda()
    aws = T.aligned_workspace(T.teno_adjoint_workspace_bytes(p), "cuda")
    mu = torch.empty_like(U)
    T.teno_rhs_vjp(p, U, U.clone(), mu, None, aws)
    done("adjoint", aws, bool(torch.isfinite(mu).all()))
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    _child()
