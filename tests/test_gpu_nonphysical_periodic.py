"""The non-physical count of a periodic axis without a decision record: face n is
face 0's image and is not counted again, whichever launch computes it, so the
count does not depend on where along the axis the non-physical cell lies.  A
cell of large negative energy counts as itself and with both its faces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2109_14340_gb300 as T  # noqa: E402

# 1D sizes about the tiles of the fused stage (31 cells, overlapping by a face) and
# one that takes the four kernels; a 2D grid's single launch
GRIDS = [[31], [32], [62], [63], [137], [140001], [37, 29]]


@pytest.mark.parametrize("scheme", [8, 10, 12])
@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_count_is_the_same_along_the_axis(n, scheme):
    nd = len(n)
    p = T.teno_params_init(ndim=nd, n=n, dx=[1.0 / k for k in n], scheme=scheme)
    s = T.Solver(p)
    for at in (0, n[0] // 2, n[0] - 1):
        U = np.ones([nd + 2] + n[::-1])
        U[1:-1] = 0.0
        U[-1] = 2.5
        U[-1, ..., at] = -100.0
        s.rhs(torch.from_numpy(U).cuda())
        pencils = 1 if nd == 1 else n[1]
        # the cell and its two faces in x; in 2D a face in y per cell of the column
        assert s.status() == pencils * (3 if nd == 1 else 4), at
