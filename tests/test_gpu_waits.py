"""The bounded device waits: a wait that runs out (its limit set to no polls at all)
gives MIX_ETIMEOUT at the next synchronising call, ends by itself, and leaves a
context that works again after it is bound again.  Nothing here hangs or faults:
every barrier and copy waited for does complete."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def mx():
    from paper_2502_19081_gb300 import build, mix
    build.build()
    return mix


def _gives_up(mx, call):
    with pytest.raises(mx.MixError) as e:
        call()
    assert e.value.code == mx.MIX_ETIMEOUT


PROBE = """
#include "tc.cuh"
// all threads but half of the last warp may poll: the wait's verdicts, one a thread
__global__ void k_probe(int* out) {
    __shared__ __align__(8) unsigned long long bar;
    if (threadIdx.x == 0) {
        mixd::mbar_init(mixd::smem_u32(&bar), 1u);
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mixd::smem_u32(&bar)) : "memory");
    }
    __syncthreads();
    out[threadIdx.x] = mixd::mbar_wait_cta(mixd::smem_u32(&bar), 0u, threadIdx.x < 48 ? 1 << 10 : 0);
    out[64 + threadIdx.x] = mixd::mbar_wait_cta(mixd::smem_u32(&bar), 0u, 1 << 10);
}
extern "C" int probe(int* out) {
    k_probe<<<1, 64>>>(out);
    return (int)cudaDeviceSynchronize();
}
"""


def test_a_block_has_one_verdict(tmp_path):
    import torch
    from paper_2502_19081_gb300 import build
    nvcc = build.nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    src, so = tmp_path / "probe.cu", tmp_path / "libprobe.so"
    src.write_text(PROBE)
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-I",
                    build.INCLUDE, str(src), "-o", str(so)], check=True)
    out = torch.full((128,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert ctypes.CDLL(str(so)).probe(ctypes.c_void_p(out.data_ptr())) == 0
    v = out.cpu().numpy()
    assert (v[:64] == 0).all() and (v[64:] == 1).all()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("lmax", [0, 3])    # one l-triple (the second tile buffer stays empty), several
def test_tile_wait_runs_out(mx, prec, lmax):
    c = mx.open_context(I.small_fe_box(3, n_rad=5, l_max=lmax, r_core=4.0), precision=prec)
    c.forces()
    _, _, f0, _ = c.get_state()
    c.set_wait_limits(tile_polls=0)
    c.forces()
    _gives_up(mx, c.sync)
    c.set_wait_limits()
    c.bind()
    c.forces()
    assert np.array_equal(c.get_state()[2], f0)
    c.close()


@pytest.mark.parametrize("n", [200, 9000])
def test_grid_barrier_runs_out(mx, n):
    import torch
    wl = I.serve_request(4, "Si", n, 0.1, 300.0, I.serve_potentials())
    c = mx.open_context(wl, precision=mx.MIX_FP32)
    c.forces()
    x0, v0, f0, _ = c.get_state()
    c.set_wait_limits(grid_polls=0)
    c.step(1.0, 1)
    _gives_up(mx, c.sync)
    torch.cuda.synchronize()
    x1, v1 = c.x.clone(), c.v.clone()
    c.set_wait_limits()
    c.step(1.0, 3)               # the context's kernels do nothing any more
    _gives_up(mx, c.sync)
    torch.cuda.synchronize()
    assert torch.equal(c.x, x1) and torch.equal(c.v, v1)
    c.bind()
    c.set_state(x0, v0)
    c.forces()
    assert np.array_equal(c.get_state()[2], f0)
    c.close()


def test_limits_are_checked(mx):
    c = mx.open_context(I.small_fe_box(3), precision=mx.MIX_FP32)
    with pytest.raises(mx.MixError) as e:
        c.set_wait_limits(tile_polls=2 ** 31 - 1)
    assert e.value.code == mx.MIX_EINVAL
    c.close()


def test_tile_wait_in_a_batch_is_said_for_every_member_it_cost(mx):
    """A CTA that gave up goes on to other members' atoms without their tiles: each of
    them must report it, and one that does not must have the forces it has alone."""
    pots = I.serve_potentials()
    wls = [I.serve_request(50 + k, "Fe", 4000, 0.6, 300.0, pots) for k in range(3)]
    members = [mx.open_context(wl, precision=mx.MIX_FP32) for wl in wls]
    alone = [mx.open_context(wl, precision=mx.MIX_FP32) for wl in wls]
    for c in members:
        c.forces()
        c.sync()
    members[0].set_wait_limits(tile_polls=0)
    b = mx.Batch(members)
    b.set_fused(True)
    b.step(1.0, 1)
    _gives_up(mx, b.sync)
    assert b.info()["fused"]
    for k, (c, a) in enumerate(zip(members, alone)):
        a.step(1.0, 1)
        if c.stats(check=False)["status_bits"] & 32:
            continue
        assert k > 0 and np.array_equal(c.get_state()[2], a.get_state()[2])
    b.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_member_whose_front_gave_up_takes_no_part_in_a_batch(mx, prec):
    """One member gives up alone, unnoticed, and is then stepped with the others: it
    does not move and is reported; the others go as they go alone."""
    import torch
    pots = I.serve_potentials()
    wls = [I.serve_request(60 + k, "Si", 900 + 700 * k, 0.2, 1200.0, pots) for k in range(3)]
    members = [mx.open_context(wl, precision=prec) for wl in wls]
    state = [c.get_state() for c in members]
    b = mx.Batch(members)
    b.set_fused(True)
    members[1].set_wait_limits(grid_polls=0)
    members[1].set_state(*state[1][:2])
    members[1].step(1.0, 1)                 # a first list build that is given up
    members[1].set_wait_limits()
    torch.cuda.synchronize()
    x1 = members[1].x.clone()
    b.step(1.0, 25)
    _gives_up(mx, b.sync)
    assert b.info()["fused"] and torch.equal(members[1].x, x1)
    for k in (0, 2):
        a = mx.open_context(wls[k], precision=prec)
        a.step(1.0, 25)
        assert a.stats()["rebuilds"] > 1
        for u, w in zip(members[k].get_state()[:3], a.get_state()[:3]):
            assert np.array_equal(u, w)
    # bound again, it is a member like the others
    for c, s in zip(members, state):
        c.bind()
        c.set_state(*s[:2])
    b.step(1.0, 5)
    b.sync()
    a = mx.open_context(wls[1], precision=prec)
    a.step(1.0, 5)
    assert np.array_equal(members[1].get_state()[2], a.get_state()[2])
    b.close()
