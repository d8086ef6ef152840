"""The cheap kernel's contraction over the support of its 3-body coefficients: the
last non-zero index decides how many control points a pair reads (two where that
is enough, else four), so potentials that end at every index are compared with the
oracle, in float64 to the 1e-10 eV/A of every float64 comparison and in float to
1e-4 of the largest force (float sums of some 10^3 terms, 6e-8 * 30 * 10)."""
import dataclasses

import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("last", [0, 1, 2, 3, 4, 5, 6, 8])
def test_support_of_the_coefficients(orc, last):
    from paper_2502_19081_gb300 import mix
    wl = I.small_fe_box(31 + last, r_core=2.0, ramp=1.0)
    rng = np.random.default_rng(last)
    c3 = 0.05 * rng.standard_normal((8, 8, 8))
    c3 = 0.5 * (c3 + c3.transpose(1, 0, 2))
    c3[last:] = 0.0
    c3[:, last:] = 0.0
    wl = dataclasses.replace(wl, spline=dataclasses.replace(wl.spline, c3=c3))
    for prec, tol in ((mix.MIX_FP64, 1e-10), (mix.MIX_FP32, None)):
        ctx = mix.open_context(wl, precision=prec, regions=[])
        x, _, f, _ = ctx.get_state()
        model = orc.Model(dataclasses.replace(wl, regions=[]))
        ref, _, _ = model.forces(x, orc.MODE_METHOD)
        err = np.abs(f[:, :3] - ref[:, :3]).max()
        assert err < (tol if tol is not None else 1e-4 * np.abs(ref).max())
        ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("atoms", [25, 29, 33])
def test_half_warps_with_more_neighbours_than_their_table(orc, atoms):
    """A dense spot in a bcc bulk, whose cheap kernel runs half warps: 24 to 32
    three-body neighbours do not fit a half warp's table and go to the whole warp (the
    oracle's forces, float64, 1e-10 of the largest force of the spot), one more is an
    overflow."""
    from paper_2502_19081_gb300 import mix
    wl = I.small_fe_box(5, nx=8, ny=8, nz=8, r_core=2.0, ramp=1.0, vacancy=False)
    s = wl.system
    ctx = mix.open_context(wl, precision=mix.MIX_FP64, nbr_cap=192, regions=[])
    assert ctx.info()["cheap_lanes"] == 16
    x, v, _, _ = ctx.get_state()
    # atoms of the spot on a small sphere about its first: every one a neighbour of it
    k = np.arange(1, atoms)
    z = 1 - (2 * k - 1) / (atoms - 1)
    ph = k * np.pi * (3 - 5 ** 0.5)
    r = 1.5
    pts = np.concatenate([[[0, 0, 0]], r * np.stack([np.sqrt(1 - z * z) * np.cos(ph), np.sqrt(1 - z * z) * np.sin(ph), z], 1)])
    # the spot takes the place of the atoms inside it; those left over go with them
    ctr = np.array([0.37, 0.41, 0.46]) * s.box_len
    dist = np.sum((x[:, :3] - ctr) ** 2, axis=1)
    x2 = x.copy()
    x2[np.argsort(dist)[:atoms], :3] = ctr + pts
    ctx.set_state(x2, v)
    n3 = [int(((d2 := np.sum((x2[:, :3] - p) ** 2, axis=1)) < wl.spline.r_cut3 ** 2).sum()) - 1 for p in ctr + pts]
    if max(n3) > 32:
        with pytest.raises(mix.MixError) as e:
            ctx.forces()
            ctx.sync()
        assert e.value.code == mix.MIX_EOVERFLOW
    else:
        assert max(n3) >= 24
        ctx.forces()
        x3, _, f, _ = ctx.get_state()
        assert ctx.info()["cheap_lanes"] == 16
        import dataclasses as dc
        ref, _, _ = orc.Model(dc.replace(wl, regions=[])).forces(x3, orc.MODE_METHOD)
        assert np.abs(f[:, :3] - ref[:, :3]).max() < 1e-10 * max(1.0, np.abs(ref).max())
    ctx.close()
