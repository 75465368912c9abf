"""What the library's host code does when the CUDA runtime refuses: libbri.so on tests/fake_cudart.cpp (device memory is
host memory of a limited size, kernels only leave their names), each test in a process of its own, no GPU."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
INCLUDE = "/usr/local/cuda/include"
OOM, CUDA, NOLINKS = -3, -2, -4

PREAMBLE = """
import ctypes, sys
sys.path.insert(0, {root!r})
fake = ctypes.CDLL({fake!r})
fake.fake_launched.restype = ctypes.c_char_p
for f in ("fake_pool_kept", "fake_pool_kept_on", "fake_largest", "fake_default_threshold"):
    getattr(fake, f).restype = ctypes.c_size_t
fake.fake_memory_left.argtypes = [ctypes.c_size_t]
from paper_1701_00726_gb300 import _lib
lib = _lib.load()
P = ctypes.c_void_p

def lattice(*dims):
    h = P()
    assert lib.bri_create(ctypes.byref(h), (ctypes.c_int * 4)(*dims), 0, P(16)) == 0
    return h

def device(n):
    p = P()
    assert fake.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(n)) == 0
    return p

def launched():
    out = [fake.fake_launched(i).decode() for i in range(fake.fake_launches())]
    fake.fake_forget()
    return out
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(INCLUDE, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    from paper_1701_00726_gb300 import _lib, build
    if shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc"):
        build.build()
    elif not os.path.exists(_lib.LIB_PATH):
        pytest.skip("no CUDA toolkit to build libbri.so")
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run([gxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", INCLUDE, "-o", so,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp")], check=True)

    def go(body):
        code = PREAMBLE.format(root=ROOT, fake=so) + textwrap.dedent(body)
        res = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LD_PRELOAD=so), capture_output=True, text=True,
                             timeout=300)
        assert res.returncode == 0, res.stdout + res.stderr

    return go


@pytest.mark.parametrize("first,second", [(0.0, 1.0), (1.0, 1.0), (1.0, 0.0)])
def test_failed_rebuild_of_the_links(run, first, second):
    """Without memory for what a rebuild needs nothing of the links of the last one is overwritten (no kernel runs, the
    same operator answers); a launch that fails in the middle of one leaves a context that refuses to compute."""
    run(f"""
    h, V = lattice(6, 5, 4, 3), 360
    u, x, y = device(V * 576), device(V * 96), device(V * 96)
    assert lib.bri_build_links(h, u, {first}) == 0
    fake.fake_forget()
    assert lib.bri_apply(h, y, x, 1, -1.0, 0, 1) == 0 and lib.wils_apply(h, y, x, 1, -1.0, 0, 1) == 0
    before = launched()
    if {second}:
        fake.fake_memory_left(V * 1000)  # less than the transient two-hop paths
        assert lib.bri_build_links(h, u, {second}) == {OOM}
        assert launched() == []
        assert lib.bri_apply(h, y, x, 1, -1.0, 0, 1) == 0 and lib.wils_apply(h, y, x, 1, -1.0, 0, 1) == 0
        assert launched() == before
        fake.fake_memory_left(1 << 40)
    fake.fake_launch_error(98)
    assert lib.bri_build_links(h, u, {second}) == {CUDA}
    fake.fake_launch_error(0)
    assert lib.bri_apply(h, y, x, 1, -1.0, 0, 1) == {NOLINKS} and lib.wils_apply(h, y, x, 1, -1.0, 0, 1) == {NOLINKS}
    assert lib.bri_build_links(h, u, {second}) == 0 and lib.bri_apply(h, y, x, 1, -1.0, 0, 1) == 0
    """)


@pytest.mark.parametrize("nrhs,prec", [(1, 1), (3, 2), (40, 1)])
def test_large_fp32_application_without_scratch(run, nrhs, prec):
    """Under capture an application leaves kernels only in the caller's graph (an allocation node would bar it from child
    graphs, conditional bodies and a second instantiation), and without memory for packed spinors it runs all the same:
    one launch, nothing allocated."""
    run(f"""
    h, V = lattice(10, 9, 10, 11), 9900
    u, x, y = device(V * 576), device(V * 96 * {nrhs}), device(V * 96 * {nrhs})
    assert lib.bri_build_links(h, u, 0.0) == 0
    for setting in ("capture", "memory"):
        fake.fake_forget()
        fake.fake_largest()
        (fake.fake_capturing if setting == "capture" else fake.fake_memory_left)(1 if setting == "capture" else 0)
        assert lib.bri_apply(h, y, x, {nrhs}, -1.0, 0, {prec}) == 0
        assert fake.fake_largest() == 0
        kernels = launched()
        assert len(kernels) == 1 and "bri_pair_kernel" in kernels[0], kernels
        fake.fake_capturing(0)
    """)


def test_memory_kept_between_calls(run):
    """Operator calls and link constructions leave at most 1 GiB of scratch in a pool (the two-hop paths of 24^3 x 28 are
    1.3 GB); solver workspaces stay in the default pool of the device they ran on, on every device; the last context to
    go gives all of it back and the default pools have their thresholds again."""
    run("""
    h, V = lattice(24, 24, 24, 28), 387072
    u, x, y = device(V * 576), device(V * 192 * 2), device(V * 192 * 2)
    assert lib.bri_build_links(h, u, 1.0) == 0
    assert fake.fake_pool_kept() <= 1 << 30
    for prec in (1, 2, 3):
        assert lib.bri_apply(h, y, x, 2, -1.0, 0, prec) == 0
    fake.cudaDeviceSynchronize()
    assert fake.fake_pool_kept() <= 1 << 30 and fake.fake_default_threshold(0) == 0
    small = []
    for dev in (0, 1):
        fake.fake_device(dev)
        k = lattice(10, 9, 10, 11)
        small.append(k)
        assert lib.bri_build_links(k, u, 1.0) == 0
        st = _lib.BriStats()
        st.maxiter = 8
        assert lib.sign_apply_multishift(k, y, x, 1, 4, 0, 1.0, 1.0, 1e-3, 0, ctypes.byref(st)) >= 0
        assert fake.fake_default_threshold(dev) > 1 << 40 and fake.fake_pool_kept_on(dev) > 0
    for k in small:
        lib.bri_destroy(k)
    assert fake.fake_pool_kept_on(1) > 0
    fake.fake_device(0)
    lib.bri_destroy(h)
    for dev in (0, 1):
        assert fake.fake_pool_kept_on(dev) == 0 and fake.fake_default_threshold(dev) == 0
    """)


@pytest.mark.parametrize("n,nrhs", [(1, 2), (4, 3)])
def test_mixed_solve_at_the_memory_limit(run, n, nrhs):
    """A mixed solve runs in the memory that the spinors' own layout needs: solutions 192 n, source 96, and 96 bytes for
    each of the n directions, r, t, q and the ring of four residuals, per site and right-hand side (the packed form's
    ring has eight); with a sixteenth less it is refused."""
    run(f"""
    h, V = lattice(10, 9, 10, 11), 9900
    u, x, y = device(V * 576), device(V * 192 * {nrhs}), device(V * 192 * {nrhs})
    assert lib.bri_build_links(h, u, 0.0) == 0
    assert lib.bri_apply(h, y, x, 1, -1.0, 0, 3) == 0  # the double-word links of the residuals, kept by the context
    need = V * {nrhs} * (192 * {n} + 96 + 96 * ({n} + 7))
    st = _lib.BriStats()
    st.maxiter = 8
    for left, rcs in ((need * 2, (0, 1)), (need + V * {nrhs} * 8 + 65536, (0, 1)), (need - need // 16, ({OOM},))):
        fake.fake_memory_left(left)
        assert lib.sign_apply_multishift(h, y, x, {nrhs}, {n}, 0, 1.0, 1.0, 1e-3, 1, ctypes.byref(st)) in rcs
    """)


@pytest.mark.parametrize("prec", [0, 1])
def test_flags_of_many_systems(run, prec):
    """The done flags of more systems than the context's pinned block holds (16384) go elsewhere: no copy leaves its block."""
    run(f"""
    h, V, nrhs = lattice(2, 2, 2, 2), 16, 16400
    u, x, y = device(V * 576), device(V * 192 * nrhs), device(V * 192 * nrhs)
    assert lib.bri_build_links(h, u, 0.0) == 0
    st = _lib.BriStats()
    st.maxiter = 8
    rc = lib.sign_apply_multishift(h, y, x, nrhs, 1, 0, 1.0, 1.0, 1e-3, {prec}, ctypes.byref(st))
    assert fake.fake_out_of_range() == 0 and rc >= 0, lib.bri_last_error()
    """)
