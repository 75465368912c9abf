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
