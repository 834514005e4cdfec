"""Line sweeps (several colour passes of one class of vertex lines per launch,
the smoothing of the default kernel choice) against the FP64 oracle's smoothing
step and against the block-per-patch colour passes, at the sizes where the
sweep's segments, halos and line ends can go wrong: lines of one, two and three
vertices, segments whose ends carry every colour, one block and several blocks
per line, every degree, precision and grouping of right-hand sides.

Tolerances: FP64 1e-10 relative to the oracle (as for every smoothing kernel),
2e-10 between two kernels; FP32 and BF16 inverses 2e-5 between two kernels,
twice the 1e-5 bound of the FP32 rounding model on these lognormal fields.
"""
import numpy as np
import pytest

from oracle import multigrid as mg
from paper_1602_04858_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402

# (d, k, n_coarse, n_levels)
SMALL = [(2, 0, 2, 3), (2, 0, 5, 3), (2, 1, 2, 3), (2, 1, 3, 3), (2, 1, 5, 2), (2, 1, 7, 3), (2, 2, 2, 3), (2, 2, 3, 2),
         (3, 0, 2, 3), (3, 0, 5, 2)]
LARGE = [(2, 0, 7, 6), (2, 1, 3, 6), (2, 1, 5, 5), (2, 1, 4, 6), (2, 2, 3, 5), (3, 0, 3, 4), (3, 0, 5, 3)]


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def field(d, n):
    return inputs.lognormal_c(n, d, 1.5, 2.0, 11)


def handle(case, **kw):
    d, k, n0, L = case
    return mgdarcy.Multigrid(d, n0, L, k, kw.pop("mu", 0.05), dev(field(d, n0 << (L - 1))), dense_level=0, **kw)


@pytest.mark.parametrize("mu", [0.0, 0.05])
@pytest.mark.parametrize("case", SMALL)
def test_smoothing_matches_oracle(case, mu):
    d, k, n0, L = case
    H = mg.Hierarchy(d, n0, L, k, mu, field(d, n0 << (L - 1)))
    G = handle(case, mu=mu)
    rng = np.random.default_rng(3)
    for j in range(1, L):
        n = H.levels[j].S.ndof
        x0, b = rng.standard_normal(n), rng.standard_normal(n)
        x = dev(x0)
        G.smooth(j, x, dev(b), steps=2)   # two steps: a run that spans them
        xo = mg.smooth_step(H.levels[j], mg.smooth_step(H.levels[j], x0, b), b)
        assert np.max(np.abs(x.cpu().numpy() - xo)) <= 1e-10 * np.max(np.abs(xo)), f"level {j}"
    assert G.sync(check=False) == 0


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_bf16inv"])
@pytest.mark.parametrize("case", LARGE)
def test_smoothing_matches_colour_passes(case, precision):
    L = case[3]
    G, B = handle(case, precision=precision), handle(case, precision=precision, pass_kernel=2)
    tol = 2e-10 if precision == "fp64" else 2e-5
    rng = np.random.default_rng(4)
    for j in range(1, L):
        n = G.ndof(j)
        x0, b = dev(rng.standard_normal(n)), dev(rng.standard_normal(n))
        xs, xb = x0.clone(), x0.clone()
        G.smooth(j, xs, b, steps=2)
        B.smooth(j, xb, b, steps=2)
        assert torch.linalg.norm(xs - xb).item() <= tol * torch.linalg.norm(xb - x0).item(), f"level {j}"
    assert G.sync(check=False) == 0


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nrhs", [4, 5, 9])
@pytest.mark.parametrize("case", [(2, 0, 5, 4), (2, 1, 3, 5), (2, 2, 3, 3), (3, 0, 3, 3)])
def test_grouped_right_hand_sides(case, nrhs, precision):
    """Groups of four right-hand sides and the rest one by one: every vector's
    V-cycle equals the one of a handle with a single right-hand side."""
    G, S = handle(case, precision=precision, nrhs=nrhs), handle(case, precision=precision)
    n = S.ndof()
    r = dev(np.random.default_rng(5).standard_normal((nrhs, n)))
    z, zs = torch.zeros_like(r), torch.zeros(n, dtype=torch.float64, device="cuda")
    G.vcycle(r, z)
    tol = 2e-10 if precision == "fp64" else 2e-5
    for q in range(nrhs):
        S.vcycle(r[q].contiguous(), zs)
        assert torch.linalg.norm(z[q] - zs).item() <= tol * torch.linalg.norm(zs).item()
    assert G.sync(check=False) == 0
