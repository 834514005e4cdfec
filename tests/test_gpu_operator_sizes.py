"""The 2-D FP64 operator of RT_0 on both sides of the size where it changes from
its tensor factors to the row plans (128^2 cells),
against the oracle's matrix: 128^2 and 132^2, and the residual norm of a coarser
level through the handle of a finer one, whose kernel and number of partial sums
differ.  Tolerance per row 1e-13 of |A| |x|, as for the factored rows.
"""
import numpy as np
import pytest

from oracle import multigrid as mg
from paper_1602_04858_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402


@pytest.mark.parametrize("n0,levels", [(8, 5), (33, 3)], ids=["128", "132"])
def test_both_sides_of_the_size_rule(n0, levels):
    c = inputs.lognormal_c(n0 << (levels - 1), 2, 1.5, 3.0, 7)
    H = mg.Hierarchy(2, n0, levels, 0, 0.3, c)
    G = mgdarcy.Multigrid(2, n0, levels, 0, 0.3, torch.as_tensor(c, device="cuda"), precision="fp64", dense_level=0)
    rng = np.random.default_rng(n0)
    for j, L in enumerate(H.levels):
        x, b = rng.standard_normal((2, L.S.ndof))
        xd, bd = torch.as_tensor(x, device="cuda"), torch.as_tensor(b, device="cuda")
        y, r = torch.zeros_like(xd), torch.zeros_like(xd)
        G.apply(xd, y, level=j)
        ref = L.A @ x
        bound = 1e-13 * (abs(L.A) @ np.abs(x)) + 1e-300
        assert np.all(np.abs(y.cpu().numpy() - ref) <= bound)
        norm = G.residual_norm(xd, bd, r, level=j)
        res = b - ref
        assert np.all(np.abs(r.cpu().numpy() - res) <= bound + 1.2e-16 * np.abs(res))
        assert abs(norm - np.linalg.norm(res)) <= 1e-13 * np.linalg.norm(res) * L.S.ndof ** 0.5
