"""A grid that takes the single launch, in a workspace of exactly the size asked
for: right-hand side, step, recording step and frozen replays leave the bytes
behind it alone, and the replay gives the recorded result."""
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T  # noqa: E402

CASES = {
    "1d-s8": lambda: workloads.riemann_1d(137, scheme=8),
    "1d-limiter-s10": lambda: dict(workloads.double_rarefaction_1d(400, scheme=10), limiter=1),
    "2d-limiter-s12": lambda: dict(workloads.quadrants_2d(37, 29, scheme=12), limiter=1),
    "2d-s10": lambda: workloads.quadrants_2d(128, 128, scheme=10),
    "3d-s8": lambda: workloads.tgv_3d(13, scheme=8),
}


@pytest.mark.parametrize("name", CASES)
def test_stays_inside(name):
    c = CASES[name]()
    p = T.teno_params_init(ndim=c["ndim"], n=c["n"], dx=c["dx"], scheme=c["scheme"], gamma=c["gamma"],
                           bc_lo=c["bc_lo"], bc_hi=c["bc_hi"], limiter=c.get("limiter", 0))
    size, guard = T.teno_workspace_bytes(p), 4 << 20
    assert size % 8 == 0
    room = torch.zeros(size + guard, dtype=torch.uint8, device="cuda")
    assert room.data_ptr() % 256 == 0
    room[size:] = 0xA5
    ws = room[:size]
    U = torch.from_numpy(c["U"].copy()).cuda()
    dt = 1e-5
    fl = torch.zeros(T.teno_flags_bytes(p), dtype=torch.uint8, device="cuda")
    rec, plain, frozen = (torch.empty_like(U) for _ in range(3))
    T.teno_rhs(p, U, rec, dt, fl, ws)
    T.teno_rhs(p, U, plain, dt, None, ws)
    T.teno_rhs_frozen(p, U, frozen, fl, ws, dt)
    assert torch.equal(rec, plain)
    # the frozen coefficients are the recorded stencils' linear schemes: each flux to some
    # ten roundings of 2^-53, over dx as the result itself
    assert float((frozen - rec).abs().max()) <= 1e-13 * float(rec.abs().max())
    steps = torch.zeros(3 * fl.numel(), dtype=torch.uint8, device="cuda")
    Ur, U1, U2 = U.clone(), torch.empty_like(U), torch.empty_like(U)
    T.teno_rk3_step_record(p, Ur, dt, U1, U2, steps, ws)
    Uf, Up = U.clone(), U.clone()
    T.teno_rk3_step_frozen(p, Uf, dt, steps, ws)
    T.teno_rk3_step(p, Up, dt, None, ws)
    assert torch.equal(Ur, Up)
    assert torch.equal(room[size:], torch.full_like(room[size:], 0xA5))
