"""The 2-D FP64 operator by its tensor factors, at the edges of its blocks.

A warp takes 30 cells along x, a block 14 along y, and the first two of either only
hand over their share: meshes of one block, of exactly one more cell, and of two,
for every degree, against the oracle's matrix; constrained rows, and the residual
with and without its vector.  Tolerance per row 1e-13 of |A| |x| (about 60 products
and sums of 1.1e-16, in any order).
"""
import numpy as np
import pytest

from oracle import multigrid as mg
from paper_1602_04858_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402


@pytest.mark.parametrize("k,n0,levels", [(0, 2, 2), (0, 7, 2), (0, 15, 2), (0, 4, 4), (1, 2, 2), (1, 7, 2), (1, 15, 2),
                                         (1, 4, 4), (2, 2, 2), (2, 7, 2), (2, 4, 4)])
def test_rows_at_block_edges(k, n0, levels):
    c = inputs.lognormal_c(n0 << (levels - 1), 2, 1.5, 3.0, 7)
    H = mg.Hierarchy(2, n0, levels, k, 0.3, c)
    G = mgdarcy.Multigrid(2, n0, levels, k, 0.3, torch.as_tensor(c, device="cuda"), precision="fp64", dense_level=0)
    rng = np.random.default_rng(n0)
    for j, L in enumerate(H.levels):
        x, b = rng.standard_normal((2, L.S.ndof))
        xd, bd = torch.as_tensor(x, device="cuda"), torch.as_tensor(b, device="cuda")
        y, r = torch.zeros_like(xd), torch.zeros_like(xd)
        G.apply(xd, y, level=j)
        bound = 1e-13 * (abs(L.A) @ np.abs(x)) + 1e-300
        ref = L.A @ x
        assert np.all(np.abs(y.cpu().numpy() - ref) <= bound)
        assert np.array_equal(y.cpu().numpy()[L.cm], x[L.cm])
        norm = G.residual_norm(xd, bd, r, level=j)
        res = b - ref
        assert np.all(np.abs(r.cpu().numpy() - res) <= bound + 1.2e-16 * np.abs(res))
        want = np.linalg.norm(res)
        assert abs(norm - want) <= 1e-13 * want * L.S.ndof ** 0.5
        assert G.residual_norm(xd, bd, level=j) == norm
