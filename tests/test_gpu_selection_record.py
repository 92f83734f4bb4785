"""The C_T exponent bits of a selection-only record (teno_rk3_step_record_sel):
zero only where the recorded selection holds at every exponent the parameters
allow, the exponent itself wherever it decided.  alpha_1 = 14, alpha_2 = 6.4
allow 7 .. 14, and the selection is monotone in C_T = 10^-n, so a zero byte
must hold the selection of a run with the exponent fixed at 7 (alpha_1 = 7,
alpha_2 = 0); any other byte equals the full record's."""
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

# both launch forms (one launch, four kernels) of a 2D and a 3D grid
CASES = {
    "2d-one-launch-s8": lambda: workloads.adjoint_2d(40, 32, scheme=8),
    "2d-four-kernels-s10": lambda: workloads.adjoint_2d(260, 200, scheme=10),
    "3d-one-launch-s12": lambda: workloads.tgv_3d(12, scheme=12),
    "3d-four-kernels-s10": lambda: workloads.tgv_3d(22, scheme=10),
}


@pytest.mark.parametrize("name", CASES)
def test_exponent_bits(name):
    c = CASES[name]()
    kw = dict(ndim=c["ndim"], n=c["n"], dx=c["dx"], scheme=c["scheme"], gamma=c["gamma"],
              bc_lo=c["bc_lo"], bc_hi=c["bc_hi"])
    p = T.teno_params_init(**kw)
    s = T.Solver(p)
    U0 = torch.from_numpy(np.ascontiguousarray(c["U"])).cuda()
    ndec, flb = T.record_layout(p)[1], T.teno_flags_bytes(p)
    full = s.rhs(U0, flags=True)[1][:ndec].cpu().numpy()
    at7 = T.Solver(T.teno_params_init(ct_alpha1=7.0, ct_alpha2=0.0, **kw)).rhs(U0, flags=True)[1]
    at7 = at7[:ndec].cpu().numpy()
    dt, _, _ = oracle.cfl_dt(oracle_params(c), c["U"], 0.4)
    U, U1, U2 = U0.clone(), torch.empty_like(U0), torch.empty_like(U0)
    fl = torch.empty(3 * flb, dtype=torch.uint8, device="cuda")
    T.teno_rk3_step_record_sel(p, U, dt, U1, U2, fl, s.ws)
    sel = fl[:ndec].cpu().numpy()                        # of L(U0)
    zero = (sel >> 5) == 0
    assert zero.any() and not zero.all()
    assert np.array_equal(sel[~zero], full[~zero])
    assert np.array_equal(sel[zero] & 31, full[zero] & 31)
    assert np.array_equal(sel[zero] & 31, at7[zero] & 31)
    # the exponent does decide in this state: some selections differ at 7
    assert np.count_nonzero((full & 31) != (at7 & 31)) > 0
