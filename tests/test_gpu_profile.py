"""The phases of a profiled evaluation: the first three are parts of one kernel, and the
part of the lists is there when they are rebuilt and zero when they are not."""
import pytest

from paper_2502_19081_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("rule", [False, True])
def test_list_phase_only_when_rebuilding(rule):
    from paper_2502_19081_gb300 import mix
    wl = I.serve_request(3, "Si", 6000, 0.05, 300.0, I.serve_potentials())
    c = mix.open_context(wl, precision=mix.MIX_FP32)
    if rule:
        c.set_seed_rule(2.9, 0.0, 3.0, 5, 5.0, 5.0)
    x, v, _, _ = c.get_state()
    c.profile(True)
    c.set_state(x, v)
    c.forces()
    tot0, first, n0 = c.get_profile()
    assert n0 == 1 and (first > 0).all()
    c.forces()
    tot1, second, n1 = c.get_profile()
    assert n1 == 2 and second[1] == 0.0 and second[0] > 0 and second[2] > 0
    assert abs(tot1 - tot0 - second).max() < 1e-6
    c.profile(False)
    c.step(1.0, 2)
    c.profile(True)
    c.step(1.0, 1)          # a captured step
    assert (c.get_profile()[1][[0, 2, 3, 4, 5]] > 0).all()
    c.close()
