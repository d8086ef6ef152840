"""Members of a tuned batch that are evaluated one after the other (new regions) open
their evaluations with every block that is resident, whatever divisor the tuning
chose for members that step side by side.  A stand-in for the runtime's cooperative
launch, linked in front of it, notes the blocks of the last launch."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include <cuda_runtime.h>
static int g_blocks = 0;
extern "C" int shim_blocks() { return g_blocks; }
extern "C" cudaError_t __real_cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t);
extern "C" cudaError_t __wrap_cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** a, size_t m,
                                                          cudaStream_t s) {
    g_blocks = (int)g.x;
    return __real_cudaLaunchCooperativeKernel(f, g, b, a, m, s);
}
"""

CHILD = """
import sys
sys.path.insert(0, {root!r})
from paper_2502_19081_gb300 import inputs as I, mix
mix.LIB_PATH = {lib!r}
blocks = mix.lib().shim_blocks
pots = I.serve_potentials()
wls = [I.serve_request(5 + k, "Si", 1000, 0.2, 600.0, pots) for k in range(24)]
cs = [mix.open_context(wl, precision=mix.MIX_FP32) for wl in wls]
for c in cs:
    c.forces()
    alone = blocks()
b = mix.Batch(cs)
div = b.tune(reps=2)
share = [c.info()["buffer_grid"] for c in cs]
for c, wl in zip(cs, wls):
    c.set_regions(wl.regions)
b.step(1.0, 1)     # evaluates the members, then one fused step without a cooperative launch
b.sync()
assert b.info()["fused"]
assert blocks() == alone, (blocks(), alone, div)
assert [c.info()["buffer_grid"] for c in cs] == share
print("ok")
"""


def test_members_evaluated_alone_take_the_whole_front(tmp_path):
    from paper_2502_19081_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    shim, lib = tmp_path / "shim.cu", tmp_path / "libmix_blocks.so"
    shim.write_text(SHIM)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-Xlinker",
                    "--wrap=cudaLaunchCooperativeKernel", "-o", str(lib), str(shim), *objs], check=True)
    res = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, lib=str(lib))], capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr
