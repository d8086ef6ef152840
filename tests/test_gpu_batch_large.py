"""Batches of more than one front entry (512 atoms) an SM take the
front's phases as kernels of their own; from four waves of blocks on, also wider
gather chunks.  Each member's trajectory, through list rebuilds, is bit for bit
the one it has alone."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("members", [12, 13, 104])   # 144, 156 and 1,248 entries of 152; 288, 312 and 2,496 blocks of 2,432
def test_large_batch_equals_members_alone(members):
    from paper_2502_19081_gb300 import build, mix
    build.build()
    ace, spl = I.element_potentials("Si", np.random.default_rng(1), 5.0, 8, 3, 3)
    wls = [I.si_replica(70 + k, 6000 - 7 * k, "vacancy", 900.0 + 400.0 * k, ace, spl) for k in range(3)]
    alone = []
    for wl in wls:
        c = mix.open_context(wl, precision=mix.MIX_FP32)
        c.step(1.0, 25)
        assert c.stats()["rebuilds"] > 1
        alone.append(c.get_state())
        c.close()
    ctxs = [mix.open_context(wls[k % 3], precision=mix.MIX_FP32) for k in range(members)]
    b = mix.Batch(ctxs)
    b.set_fused(True)
    b.step(1.0, 25)
    b.sync()
    for k, c in enumerate(ctxs):
        x, v, f, s = c.get_state()
        xa, va, fa, sa = alone[k % 3]
        assert s == sa == 25
        assert np.array_equal(x, xa) and np.array_equal(v, va) and np.array_equal(f, fa)
    b.close()
    for c in ctxs:
        c.close()
