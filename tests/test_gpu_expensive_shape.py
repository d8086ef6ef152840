"""The float expensive kernel's block: 4 warps where the regions evaluate more atoms than
one wave of blocks of 2 holds, else 2; both give the same bits (a batch always takes 2)."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("atoms,core,threads", [(20500, 0.005, 64), (20500, 0.3, 128), (52000, 0.002, 128),
                                                (15000, 0.5, 64)])
def test_block_follows_the_evaluated_set(atoms, core, threads):
    from paper_2502_19081_gb300 import mix
    pots = {"Fe": I.element_potentials("Fe", np.random.default_rng(3), 5.5, 12, 5, 4)}
    wl = I.serve_request(3, "Fe", atoms, core, 300.0, pots)
    c = mix.open_context(wl, precision=mix.MIX_FP32)
    assert c.info()["exp_threads"] == threads
    c.step(1.0, 2)
    m = mix.open_context(wl, precision=mix.MIX_FP32)
    b = mix.Batch([m])
    b.set_fused(True)
    b.step(1.0, 2)
    b.sync()
    assert b.info()["fused"] and np.array_equal(c.get_state()[2], m.get_state()[2])
    b.close()
    if threads == 64 and atoms > 20000:      # the regions change, and the block with them
        c.set_regions([I.Region(I.REGION_SPHERE, tuple(wl.system.box_len / 2), (0.0, 0.0, 1.0), 20.0, 3.0)])
        assert c.info()["exp_threads"] == 128
        c.forces()
        c.sync()
        c.set_regions(wl.regions)
        assert c.info()["exp_threads"] == 64
    c.close()
    m.close()


@pytest.mark.gpu
def test_block_follows_the_set_of_seed_atoms():
    """Seed atoms give no size beforehand: the first synchronising call chooses."""
    from paper_2502_19081_gb300 import mix
    pots = {"Fe": I.element_potentials("Fe", np.random.default_rng(3), 5.5, 12, 5, 4)}
    wl = I.serve_request(3, "Fe", 20500, 0.005, 300.0, pots)
    c = mix.open_context(wl, precision=mix.MIX_FP32)
    for seeds, threads in ((np.arange(0, c.n, 5), 128), (np.array([100]), 64)):
        c.set_seeds(seeds, 3.0, 4.0)
        c.forces()
        c.sync()
        F = c.get_state()[2]
        assert c.stats()["n_exp"] > 2000 if threads == 128 else c.stats()["n_exp"] < 1500
        assert c.info()["exp_threads"] == threads
        c.forces()
        assert np.array_equal(F, c.get_state()[2])
        c.step(1.0, 2)
        c.sync()
        assert c.info()["exp_threads"] == threads
    c.close()
