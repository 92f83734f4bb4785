"""Decision records of an odd number of bytes: a recorded RK3 step's three
records lie back to back, so the second one's 16-bit words (the maximising
cells of the splitting speeds) then start at odd addresses.  The recorded step
must equal the plain one, its frozen replay the recorded step, and every
stage's record the record of a right-hand side on its own, bitwise."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T
import workloads


@pytest.mark.parametrize("case", [
    workloads.riemann_1d(40, scheme=10), workloads.adjoint_2d(21, 16, scheme=8),
    workloads.adjoint_2d(150, 131, scheme=8)], ids=["1d-40", "2d-21x16", "2d-150x131"])
def test_back_to_back_records_of_odd_size(case):
    p = T.teno_params_init(ndim=case["ndim"], n=case["n"], dx=case["dx"], scheme=case["scheme"],
                           gamma=case["gamma"], bc_lo=case["bc_lo"], bc_hi=case["bc_hi"])
    flb = T.teno_flags_bytes(p)
    assert flb % 2 == 1
    s = T.Solver(p)
    U = torch.from_numpy(case["U"]).cuda()
    dt = float(s.cfl_dt(U).item())
    plain, rec, again = U.clone(), U.clone(), U.clone()
    U1, U2 = torch.empty_like(U), torch.empty_like(U)
    fl = torch.zeros(3 * flb, dtype=torch.uint8, device="cuda")
    s.step(plain, dt)
    T.teno_rk3_step_record(p, rec, dt, U1, U2, fl, s.ws)
    T.teno_rk3_step_frozen(p, again, dt, fl, s.ws)
    assert torch.equal(plain, rec)
    assert torch.equal(rec, again) or (rec - again).abs().max() <= 1e-12 * rec.abs().max()
    for k, V in enumerate((U, U1, U2)):
        _, one = s.rhs(V, flags=True)
        assert torch.equal(one, fl[k * flb:(k + 1) * flb])
