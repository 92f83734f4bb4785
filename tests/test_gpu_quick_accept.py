"""The filter's first test (quick_large in csrc/teno_fast.cuh), which accepts
the largest stencil without FP64 work where no decision byte is recorded:
teno_reconstruct without flags must give bitwise the all-FP64 values.  The
stencils sit where the test's bounds are tight: a smooth wave with one value
moved until chi_p crosses C_T (bisected on the FP64 path's own choice, then
probed around it), waves whose variation is 2^-16 to 2^-24 of their size (the
test's lower limit of 2^-20 inside), and sizes across its scale limits
(2^-30, 2^50), with signs, zeros, infinities and NaN among the values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T
import workloads


def recon(scheme, v, fast, flags=False):
    p = T.teno_params_init(ndim=1, n=[16], dx=[1.0], scheme=scheme)
    out = torch.empty(v.shape[0], dtype=torch.float64, device="cuda")
    fl = torch.empty(v.shape[0], dtype=torch.uint8, device="cuda") if flags else None
    T.teno_set_decision_filter(fast)
    try:
        T.teno_reconstruct(p, v.contiguous(), out, fl)
        torch.cuda.synchronize()
    finally:
        T.teno_set_decision_filter(True)
    return (out, fl) if flags else out


@pytest.mark.parametrize("scheme", [8, 10, 12])
def test_quick_acceptance_matches_fp64(scheme):
    W, H, n = scheme, scheme // 2, 200000
    g = torch.Generator(device="cuda").manual_seed(scheme)
    R = lambda lo, hi, m=n: lo + (hi - lo) * torch.rand(m, 1, generator=g, dtype=torch.float64,  # noqa: E731
                                                        device="cuda")
    x = torch.arange(W, dtype=torch.float64, device="cuda")[None, :]
    wave = torch.sin(R(0.02, 1.0) * x + R(0, 6.3)) * 2.0 ** R(-24, 2) + R(-1, 1)
    wave = wave * 2.0 ** torch.floor(R(-34, 53))
    # one value moved; bisect its displacement until the FP64 path drops S_p
    j = torch.randint(0, W, (n, 1), generator=g, device="cuda")
    unit = torch.zeros(n, W, dtype=torch.float64, device="cuda").scatter_(1, j, 1.0)
    amp = (wave.amax(1, keepdim=True) - wave.amin(1, keepdim=True)) * torch.sign(R(-1, 1))
    code = {8: 2, 10: 3, 12: 0}[scheme]
    lo, hi = torch.zeros_like(amp), torch.ones_like(amp)
    for _ in range(30):
        mid = 0.5 * (lo + hi)
        _, fl = recon(scheme, wave + unit * (amp * mid), False, True)
        keeps = ((fl & (31 if scheme == 12 else 3)) == code)[:, None]
        lo, hi = torch.where(keeps, mid, lo), torch.where(keeps, hi, mid)
    families = [wave] + [wave + unit * (amp * lo * (1 + e)) for e in
                         (-0.5, -1e-2, -1e-3, -1e-4, -1e-6, 0.0, 1e-6, 1e-4, 1e-3, 1e-2)]
    odd = wave.clone()
    odd[torch.arange(n, device="cuda"), j[:, 0]] = torch.tensor(
        [0.0, -0.0, float("inf"), float("nan"), 1e-300, 5e-324], dtype=torch.float64,
        device="cuda")[torch.randint(0, 6, (n,), generator=g, device="cuda")]
    families.append(odd)
    for v in families:
        a, b = recon(scheme, v, True), recon(scheme, v, False)
        same = (a == b) | (torch.isnan(a) & torch.isnan(b))
        bad = (~same).nonzero().flatten()
        assert bad.numel() == 0, (bad.numel(), v[bad[0]].tolist(), a[bad[0]].item(), b[bad[0]].item())


@pytest.mark.parametrize("over", [dict(), dict(ct_cr=2.0), dict(ct_alpha1=0.5, ct_alpha2=0.0)],
                         ids=["paper", "cr-2", "ct-1"])
@pytest.mark.parametrize("case", [
    workloads.riemann_1d(517, scheme=8), workloads.riemann_1d(140000, scheme=12),
    workloads.quadrants_2d(250, 231, scheme=10)], ids=["1d-517", "1d-140000", "2d"])
def test_bit_identical_stencils(case, over):
    """Sharp initial states: most stencils hold bit-identical values (velocities at
    rest give zeros).  They are accepted by the first test only where its premise
    holds; with C_r > 1, or C_T = 1 at m = 0, they must go the whole way.  Filter on
    = filter off, bitwise, records included (NaN where a fallback keeps nothing)."""
    p = T.teno_params_init(ndim=case["ndim"], n=case["n"], dx=case["dx"], scheme=case["scheme"],
                           gamma=case["gamma"], bc_lo=case["bc_lo"], bc_hi=case["bc_hi"], **over)
    s = T.Solver(p)
    U = torch.from_numpy(case["U"]).cuda()
    on, f_on = s.rhs(U, flags=True)
    plain = s.rhs(U)
    T.teno_set_decision_filter(0)
    try:
        off, f_off = s.rhs(U, flags=True)
    finally:
        T.teno_set_decision_filter(1)
    assert torch.equal(f_on, f_off)
    for r in (on, plain):
        assert torch.equal(r.nan_to_num(7.0), off.nan_to_num(7.0))
