"""A front kernel that cannot be launched (a cooperative launch the runtime refuses) is
an error of the call that wanted it: nothing else of that evaluation runs, no graph
without it is kept, and the next call works.  The refusal comes from a stand-in for
the runtime's call, linked in front of it; the GPU sees only launches that succeed."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include <cuda_runtime.h>
static int g_refuse = 0;
extern "C" void shim_refuse(int n) { g_refuse = n; }
extern "C" cudaError_t __real_cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t);
extern "C" cudaError_t __wrap_cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** a, size_t m,
                                                          cudaStream_t s) {
    if (g_refuse > 0) {
        --g_refuse;
        return cudaErrorCooperativeLaunchTooLarge;
    }
    return __real_cudaLaunchCooperativeKernel(f, g, b, a, m, s);
}
"""

CHILD = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
from paper_2502_19081_gb300 import inputs as I, mix
mix.LIB_PATH = {lib!r}
refuse = mix.lib().shim_refuse
wls = [I.serve_request(5 + k, "Si", 700 + 300 * k, 0.2, 600.0, I.serve_potentials()) for k in range(2)]
ref = []
for wl in wls:
    c = mix.open_context(wl, precision=mix.MIX_FP32, graphs=False)
    c.step(1.0, 4)
    ref.append(c.get_state())
    c.close()

def refused(call, *args):
    refuse(1)
    try:
        call(*args)
    except mix.MixError as e:
        assert e.code == mix.MIX_ECUDA, e
    else:
        raise AssertionError("no error")
    finally:
        refuse(0)

def same(c, r):
    assert all(np.array_equal(a, b) for a, b in zip(c.get_state()[:3], r[:3]))

for graphs in (False, True):
    c = mix.open_context(wls[0], precision=mix.MIX_FP32, graphs=graphs)
    refused(c.forces)
    c.forces()
    c.sync()
    before = c.x.clone(), c.v.clone(), c.f.clone()
    refused(c.step, 1.0, 1)
    c.sync()
    assert all(torch.equal(a, b) for a, b in zip(before, (c.x, c.v, c.f)))
    assert c.get_state()[3] == 0
    c.step(1.0, 4)
    same(c, ref[0])
    refused(c.tune, 1)
    c.close()
cs = [mix.open_context(wl, precision=mix.MIX_FP32) for wl in wls]
for c in cs:
    c.forces()
b = mix.Batch(cs)
b.set_fused(False)
refused(b.step, 1.0, 1)
b.step(1.0, 4)
b.sync()
for c, r in zip(cs, ref):
    same(c, r)
print("ok")
"""


def test_refused_front_launch(tmp_path):
    from paper_2502_19081_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    shim, lib = tmp_path / "shim.cu", tmp_path / "libmix_refuse.so"
    shim.write_text(SHIM)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-Xlinker",
                    "--wrap=cudaLaunchCooperativeKernel", "-o", str(lib), str(shim), *objs], check=True)
    res = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, lib=str(lib))], capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr
