"""Device-side waits of the line sweeps that run out, made to by the host-set
limit alone: zero (every wait at once) and 100 ns (some of a launch's, in some
of its teams and blocks).  The blocks of a line go on exchanging updates and
none leaves while a neighbour still sends, so the calls end, the timeout is
reported, and with the limit restored the handle gives the same result to the
last bit.  Levels whose lines are one block and several, teams of one and three
warps, one and several right-hand sides.
"""
import numpy as np
import pytest

from paper_1602_04858_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1602_04858_gb300 import mgdarcy  # noqa: E402

TIMEOUT = 6


@pytest.mark.parametrize("nrhs", [1, 5])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_bf16inv"])
@pytest.mark.parametrize("d,k,n0,levels", [(2, 0, 4, 6), (2, 1, 4, 5), (2, 1, 7, 5), (2, 2, 4, 4), (3, 0, 3, 4)])
def test_waits_that_run_out_end_the_call(d, k, n0, levels, precision, nrhs):
    c = torch.as_tensor(inputs.lognormal_c(n0 << (levels - 1), d, 1.5, 4.0, 71), device="cuda")
    G = mgdarcy.Multigrid(d, n0, levels, k, 0.01, c, precision=precision, dense_level=0, nrhs=nrhs)
    r = torch.as_tensor(np.random.default_rng(72).standard_normal(nrhs * G.ndof()), device="cuda")
    z = torch.zeros_like(r)
    G.vcycle(r, z)
    assert G.sync(check=False) == 0
    out = torch.zeros_like(r)
    G.set_wait_limit(0.0)
    G.vcycle(r, out)
    assert G.sync(check=False) == TIMEOUT
    G.set_wait_limit(1e-7)
    for _ in range(3):
        G.vcycle(r, out)
    assert G.sync(check=False) in (0, TIMEOUT)   # whether a copy takes longer is up to the hardware
    G.set_wait_limit(2.0)
    G.vcycle(r, out)
    assert G.sync(check=False) == 0
    assert torch.equal(out, z)
