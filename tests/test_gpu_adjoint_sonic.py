"""The sign of u - c in the reverse of the splitting speed |u - c| where u and c
differ by one unit of the last place.  Three 1D states with the same densities
and sound speed c = 1 + 2^-52 in every cell and u = c - 2^-52, c, c + 2^-52:
the speed's derivative is -1, 0, +1 times the same factor, so with one and the
same decision record the vector-Jacobian products of the outer two lie on
either side of the middle one's at equal distances, up to rounding: their mean
is within 1e-9 of it (of their size; the states differ by 1e-16, the condition
of the sums is a few hundred), their difference is the factor itself, which a
rough density makes large."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T  # noqa: E402

GAMMA = 1.4
C0 = 1.0 + 2.0 ** -52


def _near(x, most=40):
    out, a, b = [x], x, x
    for _ in range(most):
        a, b = np.nextafter(a, np.inf), np.nextafter(b, -np.inf)
        out += [a, b]
    return out


def _cell(rho, u):
    """Momentum and energy whose primitives, by the library's own operations, are
    u and C0 to the last bit (None where no double gives them)."""
    rinv, gm1 = 1.0 / rho, GAMMA - 1.0
    for m in _near(rho * u, 3):
        if m * rinv != u:
            continue
        ke = 0.5 * (m * u)
        for E in _near(rho / GAMMA / gm1 * C0 * C0 + ke):
            if np.sqrt((GAMMA * (gm1 * (E - ke))) * rinv) == C0:
                return m, E
    return None


def _states(n, seed):
    g = np.random.default_rng(seed)
    us = [C0 - 2.0 ** -52, C0, C0 + 2.0 ** -52]
    cols = []
    while len(cols) < n:
        rho = float(g.uniform(0.5, 1.5))
        cells = [_cell(rho, u) for u in us]
        if all(cells):
            cols.append([(rho,) + c for c in cells])
    return [np.ascontiguousarray(np.array([c[k] for c in cols]).T) for k in range(3)]


@pytest.mark.parametrize("scheme", [8, 10, 12])
def test_sign_within_rounding(scheme):
    n = 96
    p = T.teno_params_init(ndim=1, n=[n], dx=[1.0 / n], scheme=scheme, gamma=GAMMA)
    rec = torch.zeros(T.teno_flags_bytes(p), dtype=torch.uint8, device="cuda")
    rec[:T.record_layout(p)[1]] = {8: 2, 10: 3, 12: 0}[scheme]     # S_p everywhere
    lam = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, (3, n))).cuda()
    aws = T.aligned_workspace(T.teno_adjoint_workspace_bytes(p), "cuda")
    mu = []
    for U in _states(n, 17):
        out = torch.empty(3, n, dtype=torch.float64, device="cuda")
        T.teno_rhs_vjp(p, torch.from_numpy(U).cuda(), lam, out, rec, aws)
        mu.append(out.cpu().numpy())
    size = np.abs(mu[1]).max()
    assert np.abs(mu[2] - mu[0]).max() > 1e-3 * size
    assert np.abs(0.5 * (mu[0] + mu[2]) - mu[1]).max() <= 1e-9 * size
