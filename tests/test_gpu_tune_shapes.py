"""What the tuners leave in the launch shapes of the kernel that opens an evaluation,
which also builds the lists: a batch's divisor divides what is resident, and a context
tuned alone keeps all of it."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _members(mix, n):
    pots = I.serve_potentials()
    return [mix.open_context(I.serve_request(20 + k, "Si", 2500 + 300 * k, 0.1, 900.0, pots), precision=mix.MIX_FP32)
            for k in range(n)]


def test_batch_divisor_divides_the_resident_front():
    import torch
    from paper_2502_19081_gb300 import mix
    members = _members(mix, 4)
    alone = _members(mix, 4)
    for c in members + alone:
        c.set_seed_rule(2.9, 0.0, 3.0, 5, 4.0, 4.0)     # such members step as graphs of their own
        c.forces()
    b = mix.Batch(members)
    div = b.tune(reps=2)
    resident = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    for c in members:
        assert 1 <= c.info()["buffer_grid"] <= max(1, resident // div)
    b.step(1.0, 25)
    b.sync()
    assert not b.info()["fused"]
    for c, a in zip(members, alone):
        a.step(1.0, 25)
        assert a.stats()["rebuilds"] > 1
        assert np.array_equal(c.get_state()[0], a.get_state()[0])
    b.close()


def test_tuned_alone_keeps_the_whole_front():
    from paper_2502_19081_gb300 import mix
    c = _members(mix, 1)[0]
    b = mix.Batch([c])
    b.tune(reps=1)
    c.tune(reps=2)
    assert c.info()["buffer_grid"] == 0
    b.close()
    c.close()
