"""Workspace of grids and batches that take the single launch: no queue between
kernels, only the rows a frozen replay passes from its sweep to its finish
(values and Roe states, with the limiter the cells' states and fluxes)."""
import pytest

import paper_2109_14340_gb300 as T
from helpers import tiles_of


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2109_14340_gb300 import _build
    _build.build()
    T.load()


def _base(n, scheme):
    nd, cells = len(n), 1
    for k in n:
        cells *= k
    faces = sum(cells // k * (k + 1) for k in n)
    return 8 * ((nd + 2) * (faces + cells) + (nd + 4) * cells)


# both sides of the launch rules (4096 tiles in 1D, 3072 or 1024 in 2D, 512 in 3D)
GRIDS = [([7], 8, True), ([400], 8, True), ([131000], 10, True), ([140001], 10, False),
         ([128, 128], 10, True), ([90, 88], 12, True), ([260, 200], 10, False), ([139, 133], 12, False),
         ([16, 15, 14], 12, True), ([22, 22, 22], 8, False)]


@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("n,scheme,one", GRIDS)
def test_grid(n, scheme, one, limiter):
    nd, nc = len(n), len(n) + 2
    p = T.teno_params_init(ndim=nd, n=n, dx=[0.1] * nd, scheme=scheme, limiter=limiter)
    tiles = tiles_of(dict(ndim=nd, n=n, scheme=scheme))
    rows = 8 * (2 * nc + nd + 4 + (4 * nc + 1 if limiter else 0)) * 32 * tiles
    beside = T.teno_workspace_bytes(p) - _base(n, scheme) - rows
    assert beside >= 0
    # header, counters and each part's rounding up to 256 bytes, or the queue
    assert (beside <= 16 * 256) == one


@pytest.mark.parametrize("count,one", [(200, True), (400, False)])
def test_batch(count, one):
    """Tubes of 300 cells: 10 tiles of 31 cells each, 2400 of them in one launch."""
    n = 300
    offs, total = T.pack_offsets([n] * count)
    h = T.teno_batch_create(T.teno_params_init(), [
        dict(n=n, offset=o, dx=0.01, scheme=10, limiter=1, bc_lo=1, bc_hi=1) for o in offs])
    try:
        # states, fluxes, primitives of each problem, its descriptor and its own workspace
        most = 8 * count * (3 * n + 3 * (n + 2) + 5 * n) + 256 * count + 8 * total
        assert (T.teno_batch_workspace_bytes(h) <= most + (1 << 18)) == one
    finally:
        T.teno_batch_destroy(h)
