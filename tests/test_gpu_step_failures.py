"""lbib_step when a sequence of steps cannot be captured: shorter ones take its place.
When not even single steps can be, at a context's first call, nothing is enqueued and
the next call runs.

The failure is made on the host: the library is linked once more with a wrapper
around cudaGraphInstantiate that returns an error code at the asked-for call."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WRAPPER = r"""
#include <cuda_runtime.h>
static int left = 0, failing = 0;  // calls until the failing ones, and their number
extern "C" void fail_instantiate(int after, int n) { left = after; failing = n; }
extern "C" int failures_left() { return failing; }
extern "C" cudaError_t __real_cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long);
extern "C" cudaError_t __wrap_cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long f) {
    if (failing > 0 && left-- <= 0) {
        --failing;
        return cudaErrorMemoryAllocation;
    }
    return __real_cudaGraphInstantiate(e, g, f);
}
"""


def wrapped_library(folder):
    from paper_1907_00080_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    src, lib = os.path.join(folder, "wrapper.cu"), os.path.join(folder, "liblbib_wrapped.so")
    with open(src, "w") as f:
        f.write(WRAPPER)
    subprocess.run([build._nvcc(), *build.ARCH, "-Xcompiler", "-fPIC", "-shared", "-Xlinker",
                    "--wrap=cudaGraphInstantiate", "-o", lib, src, *objs], check=True)
    return lib


def run_with_failures(path):
    """(in a process of its own: the wrapped library takes the library's place)"""
    from paper_1907_00080_gb300 import inputs, lbib
    lib = lbib.load(path)
    wl = inputs.capsule_128x32(bonds="stress")
    a, b = (lbib.Simulation(wl, precision="f32") for _ in range(2))

    def same(n):
        assert lbib.lbib_step_count(a.ctx) == lbib.lbib_step_count(b.ctx) == n
        for x, y in zip((a.populations(), a.markers(), a.bonds()), (b.populations(), b.markers(), b.bonds())):
            assert np.array_equal(x, y)

    lib.fail_instantiate(ctypes.c_int(1), ctypes.c_int(1))
    with pytest.raises(lbib.LbibError) as e:
        a.step(5)
    assert e.value.status == lbib.LBIB_E_OOM
    assert lbib.lbib_step_count(a.ctx) == 0
    for s in (a, b):
        s.step(5)  # the sequences of four steps and of one, from either buffer
    # 4 + 2 steps, of which the two cannot be captured; 8 + 2 + 1, the eight; from the
    # other buffer 4 + 2 + 1, where the four are there; and 2 x 32 with neither 32 nor 16
    for n, k in ((6, 1), (11, 0), (7, 0), (64, 0)):
        count = lbib.lbib_step_count(a.ctx)
        lib.fail_instantiate(ctypes.c_int(k), ctypes.c_int(2 if n == 64 else 1))
        a.step(n)
        assert lib.failures_left() == 0
        for _ in range(n):
            b.step(1)
        a.sync()
        b.sync()
        same(count + n)
    a.close()
    b.close()
    print("steps after failures ok")


def test_failed_captures(tmp_path):
    lib = wrapped_library(str(tmp_path))
    code = ("import sys; sys.path[:0] = [%r, %r]\nimport test_gpu_step_failures as t\nt.run_with_failures(%r)\n"
            % (ROOT, os.path.join(ROOT, "tests"), lib))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "steps after failures ok" in r.stdout
