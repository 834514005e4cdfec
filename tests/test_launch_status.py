"""Launches of the smoother on the host, with a stand-in for the CUDA runtime
(fake_cudart.cpp: two devices, kernels do not run): the shared-memory limit is
set on every device that a thread uses one after the other, whatever split it
has worked out before; a launch that fails is reported by the call and never
becomes a replayed V-cycle without it; every problem of a batch smooths as its
own pass_kernel asks; and what the line sweeps launch does not depend on the
timings of the colour passes; and small levels of RT_1 in FP64 smooth by colour
passes.  The library's own objects are linked
against the stand-in and run in a process of their own.
"""
import os
import subprocess
import sys

import pytest

from paper_1602_04858_gb300 import build as builder

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(builder.nvcc()))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    builder.build()
    out = str(tmp_path_factory.mktemp("fake") / "libmgdarcy_fake.so")
    objs = [os.path.join(builder.BUILD, o) for _, o, _ in builder.UNITS]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + os.path.join(CUDA, "include"),
                    os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-o", out], check=True, capture_output=True)
    return out


def run(lib, body):
    head = ("import ctypes, sys\nimport numpy as np\nfrom paper_1602_04858_gb300 import mgdarcy\n"
            "L = mgdarcy.load(sys.argv[1])\n"
            "L.fake_launches.restype = ctypes.c_long\n"
            "def launches(part, d=0): return L.fake_launches(d, part)\n"
            "def handle(precision='fp32', k=1, n0=4, levels=5, nrhs=1):\n"
            "    n = n0 << (levels - 1)\n"
            "    return mgdarcy.Multigrid(2, n0, levels, k, 0.01, np.ones(n * n), precision=precision, dense_level=0,\n"
            "                             nrhs=nrhs, stream=0)\n")
    r = subprocess.run([sys.executable, "-c", head + body, lib], cwd=os.path.dirname(HERE), capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("k,precision", [(0, "fp32"), (1, "fp32"), (1, "fp64"), (2, "fp32")])
def test_each_device_gets_its_limit(lib, k, precision):
    run(lib, f"""
for d in (0, 1, 0):
    L.fake_set_device(d)
    before = launches(b'k_line_sweep', d)
    G = handle({precision!r}, {k})
    r = np.zeros(G.ndof())
    G.vcycle(r, np.zeros_like(r))
    G.smooth(4, np.zeros_like(r), r)
    assert launches(b'k_line_sweep', d) > before, d
    G.close()
""")


def test_failed_launch_is_reported_and_not_replayed(lib):
    run(lib, """
G = handle()
r = np.zeros(G.ndof())
z = np.zeros_like(r)
for call in (lambda: G.vcycle(r, z), lambda: G.smooth(4, z, r)):
    L.fake_fail_launches(b'k_line_sweep')
    try:
        call()
        raise SystemExit('the failed launch was not reported')
    except mgdarcy.MGError as e:
        assert e.status == 3 and 'line sweep' in str(e), e
    L.fake_fail_launches(b'')
    before = launches(b'k_line_sweep')
    call()
    assert launches(b'k_line_sweep') > before, 'a cycle without its sweeps was replayed'
""")


def test_batch_members_smooth_as_asked(lib):
    """A problem with a forced colour-pass kernel and one left to the library, whose
    timed choice is the same kernel (every timing is equal here, so the first one
    tried), in either order: one smooths by colour passes, the other by line sweeps."""
    run(lib, """
def count(kernels):
    B = mgdarcy.Batch([dict(dim=2, n_coarse=4, n_levels=4, degree=1, mu=0.01, c=np.ones(32 * 32), precision='fp32',
                            pass_kernel=k) for k in kernels], nrhs=1, stream=0)
    r = np.zeros(B.total())
    at = launches(b'k_line_sweep'), launches(b'k_colour_pass')
    B.vcycle(r, np.zeros_like(r))
    out = launches(b'k_line_sweep') - at[0], launches(b'k_colour_pass') - at[1]
    del B
    return out
lines, none = count([0])
none2, passes = count([1])
assert lines > 0 and passes > 0 and none == none2 == 0
assert count([0, 1]) == (lines, passes)
assert count([1, 0]) == (lines, passes)
assert count([0, 0]) == (lines, 0)      # the same choice: one group, one launch for both
""")


@pytest.mark.parametrize("k,precision,nrhs", [(0, "fp32", 4), (1, "fp32", 8), (1, "fp64", 4), (1, "fp32_bf16inv", 5)])
def test_line_sweeps_do_not_follow_colour_pass_timings(lib, tmp_path, k, precision, nrhs):
    """Timings that make the colour passes' first candidate the fastest (four right-hand
    sides together) and their last one (each on its own): the same sweeps are launched."""
    for fall in (0, 1):
        run(lib, f"""
L.fake_timings_fall({fall})
G = handle({precision!r}, {k}, nrhs={nrhs})
g = ctypes.c_int()
L.mg_level_rhs_group(G.h, 4, ctypes.byref(g))
assert g.value == (1 if {fall} else 4), g.value
r = np.zeros({nrhs} * G.ndof())
at = launches(b'k_line_sweep'), launches(b'Li4ELi1EEE'), launches(b'Li1ELi1EEE')
G.vcycle(r, np.zeros_like(r))
now = launches(b'k_line_sweep') - at[0], launches(b'Li4ELi1EEE') - at[1], launches(b'Li1ELi1EEE') - at[2]
assert now[0] == now[1] + now[2] > 0, now
path = {str(tmp_path / "launches")!r}
if {fall}:
    assert open(path).read() == repr(now), now
else:
    open(path, 'w').write(repr(now))
""")


def test_small_fp64_levels_of_rt1_smooth_by_colour_passes(lib):
    """152 SMs: a colour of 32^2 has at most 11^2 patches, one right-hand side stays
    below, two do not; 40^2 has 13^2.  FP32 and RT_0 take line sweeps on every level,
    and one vector on a handle of two goes as the handle's V-cycle does."""
    run(lib, """
def swept(n0, levels, nrhs, **kw):
    G = handle(n0=n0, levels=levels, nrhs=nrhs, **kw)
    r = np.zeros(nrhs * G.ndof())
    at = launches(b'k_line_sweep')
    G.vcycle(r, np.zeros_like(r))
    v = launches(b'k_line_sweep') - at
    at = launches(b'k_line_sweep')
    G.smooth(levels - 1, np.zeros(G.ndof()), np.zeros(G.ndof()))
    return v > 0, launches(b'k_line_sweep') - at > 0
assert swept(4, 4, 1, precision='fp64') == (False, False)
assert swept(4, 4, 2, precision='fp64') == (True, True)
assert swept(5, 4, 1, precision='fp64') == (True, True)
assert swept(4, 2, 1, precision='fp64', k=0) == (True, True)
assert swept(4, 2, 1, precision='fp32') == (True, True)
""")
