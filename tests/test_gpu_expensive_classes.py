"""The float expensive kernels at the edges of their instantiation classes: n
radial functions up to 4, 8, 10, 12 and 16 (row padding, lane units, splits of
the flattened (q1, q2) index) and every lmax, i.e. every unrolled l-triple,
against the oracle.

Tolerance: a force is a sum over some 10^4 products (l-triples x n^3 x m) in
float; with unit roundoff 6e-8, random-walk growth sqrt(10^4) and a cancellation
of the terms by a factor of 10 the error stays below 6e-8 * 100 * 10 = 6e-5 of the
largest force, taken as 1e-4.  The bf16 hi/lo readout rounds each operand to
about 16 bits (1.5e-5): the same estimate gives 1.5e-5 * 10 / sqrt(10^2) of the
nu = 3 part, and the existing gate of 1e-4 relative is taken as 3e-4."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I

CASES = [(1, 2), (3, 4), (4, 6), (5, 3), (7, 5), (8, 4), (9, 4), (10, 5), (10, 6), (11, 3), (12, 6), (13, 4), (16, 3),
         (16, 6)]


def _rel_error(orc, n, lmax, precision):
    from paper_2502_19081_gb300 import mix
    wl = I.cluster_workload(100 * n + lmax, n=22, radius=5.0, n_rad=n, l_max=lmax, body_order=4)
    ctx = mix.open_context(wl, precision=precision)
    x, _, f, _ = ctx.get_state()
    ref, _, _ = orc.Model(wl).forces(x, orc.MODE_METHOD)
    ctx.close()
    return float(np.abs(f[:, :3] - ref[:, :3]).max() / np.abs(ref).max())


@pytest.mark.gpu
@pytest.mark.parametrize("n,lmax", CASES)
def test_float_forces_at_class_edges(orc, n, lmax):
    from paper_2502_19081_gb300 import mix
    assert _rel_error(orc, n, lmax, mix.MIX_FP32) < 1e-4


@pytest.mark.gpu
@pytest.mark.parametrize("n,lmax", [(3, 4), (8, 4), (9, 5), (10, 4), (12, 5), (12, 6)])
def test_split_readout_at_class_edges(orc, n, lmax):
    from paper_2502_19081_gb300 import mix
    assert _rel_error(orc, n, lmax, mix.MIX_BF16_SPLIT) < 3e-4
