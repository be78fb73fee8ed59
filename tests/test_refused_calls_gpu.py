"""Sweeps go on where the CUDA runtime refuses what makes them fast.  The library is
linked once more with a source file compiled so that one runtime call goes to a stand-in
that refuses it from the n-th call on (no fault reaches the GPU: nothing is launched or
captured by a refused call); the chain and the series must be those of the library as it
is, bit for bit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "tests", "_build")

STAND_IN = """
#include <cstdlib>
#include <cuda_runtime.h>
static bool refused()
{
    static int calls = 0;
    return calls++ >= std::atoi(std::getenv("REFUSE_FROM"));
}
extern "C" cudaError_t standin_launch(const void* f, dim3 g, dim3 b, void** a, size_t m,
                                      cudaStream_t s)
{
    return refused() ? cudaErrorCooperativeLaunchTooLarge
                     : cudaLaunchCooperativeKernel(f, g, b, a, m, s);
}
extern "C" cudaError_t standin_capture(cudaStream_t s, cudaStreamCaptureMode m)
{
    return refused() ? cudaErrorMemoryAllocation : cudaStreamBeginCapture(s, m);
}
"""

RUN = """
import ctypes, sys
lib = sys.argv[1]
if lib:
    load = ctypes.CDLL
    ctypes.CDLL = lambda path, *a, **k: load(lib if path.endswith("libspinmc.so") else path, *a, **k)
import torch
import numpy as np
from paper_1107_5463_gb300 import spinmc
d, L, n, calls = int(sys.argv[2]), int(sys.argv[3]), int(sys.argv[4]), eval(sys.argv[5])
lat = spinmc.Lattice(d, L, n=n, seed=4)
out = []
for k in calls:
    E, m = lat.sweep_series(0.4, k, 9)
    out += [E.cpu().numpy(), m.cpu().numpy()]
assert lat.state()[1] == sum(calls)
np.savez(sys.argv[6], *out, lat.get_spins())
"""


@pytest.fixture(scope="module")
def libraries():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import build
    objects = {os.path.basename(s)[:-3]: os.path.join(build.OUT, os.path.basename(s)[:-3] + ".o")
               for s in build._sources()}
    if not all(os.path.exists(o) for o in objects.values()):
        build.build(force=True)
    os.makedirs(OUT, exist_ok=True)
    base = [build.nvcc()] + build.ARCH

    def obj(src, name, extra=()):
        o = os.path.join(OUT, name + ".o")
        subprocess.run(base + build.FLAGS + list(extra) + ["-c", src, "-o", o], check=True)
        return o

    src = os.path.join(OUT, "standin.cu")
    with open(src, "w") as f:
        f.write(STAND_IN)
    standin = obj(src, "standin")
    libs = {}
    for name, define in (("ising_res", "-DcudaLaunchCooperativeKernel=standin_launch"),
                         ("lattice", "-DcudaStreamBeginCapture=standin_capture")):
        objs = [o for s, o in objects.items() if s != name]
        objs += [standin, obj(os.path.join(build.CSRC, name + ".cu"), name, [define])]
        libs[name] = os.path.join(OUT, "libspinmc_refused_%s.so" % name)
        subprocess.run(base + ["-shared", "-o", libs[name]] + objs + ["-cudart", "static"],
                       check=True)
    return libs


@pytest.mark.parametrize("source,start,d,L,n,calls", [
    ("ising_res", 0, 2, 136, 1, [4, 1]), ("ising_res", 0, 2, 1000, 1, [4, 1]),
    ("ising_res", 0, 3, 64, 1, [4, 1]), ("ising_res", 1, 2, 136, 1, [1100, 3]),
    ("lattice", 0, 2, 128, 2, [5, 40, 5]), ("lattice", 1, 2, 128, 2, [5, 40, 5]),
    ("lattice", 2, 3, 10, 3, [5, 40, 5])])
def test_the_chain_goes_on(libraries, tmp_path, source, start, d, L, n, calls):
    import numpy as np
    got = []
    for lib in ("", libraries[source]):
        out = str(tmp_path / ("out%d.npz" % len(got)))
        env = dict(os.environ, REFUSE_FROM=str(start))
        r = subprocess.run([sys.executable, "-c", RUN, lib, str(d), str(L), str(n), repr(calls),
                            out], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        with np.load(out) as z:
            got.append([z[k] for k in z.files])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
