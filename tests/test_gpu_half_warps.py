"""Half warps of the cheap kernel beside atoms with more three-body neighbours than a
half warp's table holds: the limit an overflow names, and the batched kernel, where the
two halves of a warp may belong to two systems with tables of their own."""
import dataclasses

import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _dense_spot(ctx, wl, atoms, centre):
    """The context's state with `atoms` atoms on and in a sphere of 1.5 A about a point."""
    x, v, _, _ = ctx.get_state()
    k = np.arange(1, atoms)
    z = 1 - (2 * k - 1) / (atoms - 1)
    ph = k * np.pi * (3 - 5 ** 0.5)
    q = np.sqrt(1 - z * z)
    pts = np.concatenate([[[0, 0, 0]], 1.5 * np.stack([q * np.cos(ph), q * np.sin(ph), z], 1)])
    ctr = np.asarray(centre) * wl.system.box_len
    x2 = x.copy()
    x2[np.argsort(np.sum((x[:, :3] - ctr) ** 2, axis=1))[:atoms], :3] = ctr + pts
    d = x2[:, None, :3] - x2[None, :, :3]
    d -= wl.system.box_len * np.rint(d / wl.system.box_len)
    n3 = (np.sum(d * d, axis=2) < wl.spline.r_cut3 ** 2).sum(axis=1) - 1
    return x2, v, int(n3.max())


def test_overflow_names_the_limit():
    from paper_2502_19081_gb300 import mix
    wl = I.small_fe_box(5, nx=8, ny=8, nz=8, r_core=2.0, ramp=1.0, vacancy=False)
    ctx = mix.open_context(wl, precision=mix.MIX_FP32, nbr_cap=192, regions=[])
    assert ctx.info()["cheap_lanes"] == 16
    x, v, most = _dense_spot(ctx, wl, 36, (0.37, 0.41, 0.46))
    assert most > 32
    ctx.set_state(x, v)
    with pytest.raises(mix.MixError) as e:
        ctx.forces()
        ctx.sync()
    assert e.value.code == mix.MIX_EOVERFLOW
    assert f"three-body neighbours {most} exceed 32" in str(e.value)
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shared", [True, False])
def test_batched_retake(prec, shared):
    """Two members with a spot of 25 to 32 three-body neighbours, at different places of
    their lists, and one without; forces bit for bit those of each alone."""
    from paper_2502_19081_gb300 import mix
    wls, states = [], []
    for k, (atoms, centre) in enumerate([(0, None), (27, (0.37, 0.41, 0.46)), (30, (0.13, 0.81, 0.22))]):
        wl = I.small_fe_box(5 + k, nx=8 + k, ny=8, nz=7 + k, r_core=2.0, ramp=1.0, vacancy=k == 1)
        if k and shared:
            wl = dataclasses.replace(wl, spline=wls[0].spline)
        elif k:
            wl = dataclasses.replace(wl, spline=dataclasses.replace(wl.spline, c2=wl.spline.c2 * (1.0 + 0.1 * k)))
        ctx = mix.open_context(wl, precision=prec, nbr_cap=192)
        assert ctx.info()["cheap_lanes"] == 16
        if atoms:
            x, v, most = _dense_spot(ctx, wl, atoms, centre)
            assert 24 < most <= 32
        else:
            x, v = ctx.get_state()[:2]
        wls.append(wl)
        states.append((x, v * 0.0))
        ctx.close()

    def opened():
        out = []
        for wl, s in zip(wls, states):
            c = mix.open_context(wl, precision=prec, nbr_cap=192)
            c.set_state(*s)
            out.append(c)
        return out

    dt = 1e-3    # the spot flies apart: the counts stay those of the start
    alone = opened()
    for c in alone:
        c.step(dt, 2)
        c.sync()
        assert c.info()["cheap_lanes"] == 16
    members = opened()
    b = mix.Batch(members)
    b.set_fused(True)
    b.step(dt, 2)
    b.sync()
    assert b.info()["fused"]
    for c, a in zip(members, alone):
        assert c.info()["cheap_lanes"] == 16
        for u, w in zip(c.get_state()[:3], a.get_state()[:3]):
            assert np.array_equal(u, w)
    b.close()
