"""Race detection for the line sweeps (the smoothing of the default kernel
choice), which a cap on the grid turns off, so that the comparison with one
block walking a colour does not reach them.

A patch's arithmetic depends neither on the block, team and buffer that takes
it nor on what runs beside it, so a smoothing step or a V-cycle repeated from
the same vectors must be equal to the last bit: a residual overwritten while a
slower warp of its team still reads it, a strip read while a neighbour block
writes it, or an inverse replaced too early would change bits.  Teams of
several warps (RT_2) are repeated most.  With one, two and three right-hand
sides the same patches are split differently over blocks, teams and buffers (the
lines of a launch are counted over the right-hand sides, each on its own):
every vector must still equal the single one.
"""
import numpy as np
import pytest

from paper_1602_04858_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def handle(d, k, n0, levels, precision, nrhs=1):
    c = dev(inputs.lognormal_c(n0 << (levels - 1), d, 2.0, 4.0, 91))
    return mgdarcy.Multigrid(d, n0, levels, k, 0.01, c, precision=precision, dense_level=0, nrhs=nrhs)


@pytest.mark.parametrize("precision", ["fp32", "fp32_bf16inv"])
@pytest.mark.parametrize("n0,levels", [(4, 4), (4, 5), (4, 6), (5, 5)], ids=["32", "64", "128", "80"])
def test_teams_of_several_warps_repeat_bit_for_bit(n0, levels, precision):
    rng = np.random.default_rng(92)
    for nrhs in (1, 4):
        G = handle(2, 2, n0, levels, precision, nrhs)
        r = dev(rng.standard_normal(nrhs * G.ndof()))
        x0, b = dev(rng.standard_normal(G.ndof())), dev(rng.standard_normal(G.ndof()))
        z, x = torch.zeros_like(r), x0.clone()
        G.vcycle(r, z)
        G.smooth(levels - 1, x, b, steps=2)
        assert torch.isfinite(z).all().item() and not torch.equal(x, x0)
        for rep in range(50):
            z1, x1 = torch.zeros_like(r), x0.clone()
            G.vcycle(r, z1)
            G.smooth(levels - 1, x1, b, steps=2)
            assert torch.equal(z1, z), (nrhs, rep, "V-cycle")
            assert torch.equal(x1, x), (nrhs, rep, "smoothing")
        assert G.sync(check=False) == 0


# RT_2 in FP64 smooths by colour passes, whose kernel is timed for each handle, and so do
# small levels of RT_1 in FP64 with few right-hand sides: those are compared with themselves
SPLITS = [(case, precision) for case in [(2, 0, 7, 6), (2, 1, 4, 6), (2, 1, 3, 5), (2, 2, 3, 5), (3, 0, 2, 5), (3, 0, 3, 4)]
          for precision in ("fp64", "fp32", "fp32_bf16inv") if not (case[1] == 2 and precision == "fp64")]


@pytest.mark.parametrize("case,precision", SPLITS)
def test_splits_agree_bit_for_bit(case, precision):
    d, k, n0, levels = case
    one = handle(d, k, n0, levels, precision)
    n = one.ndof()
    r = dev(np.random.default_rng(93).standard_normal(n))
    z = torch.zeros_like(r)
    one.vcycle(r, z)
    for nrhs in (1, 2, 3):
        G = handle(d, k, n0, levels, precision, nrhs)
        for rep in range(5):
            zs = torch.zeros((nrhs, n), dtype=torch.float64, device="cuda")
            G.vcycle(r.repeat(nrhs), zs)
            if rep == 0 and k == 1 and precision == "fp64":
                z = zs[0].clone()
            for q in range(nrhs):
                assert torch.equal(zs[q], z), (nrhs, rep, q)
        assert G.sync(check=False) == 0
