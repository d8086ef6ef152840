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
