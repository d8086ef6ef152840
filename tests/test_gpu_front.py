"""The one-launch front of an evaluation (integration, lists, weights, sets and
their compaction) at the sizes where its chunks can go wrong: fewer atoms than a
warp, chunk edges, empty trailing chunks, both sides of the size at which every
CTA counts the flags itself (32,768 atoms), and of the one at which it scans the
cell counts itself (8,192 cells).  Everything compared is an integer, so equality
is exact."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I


def _workload(kind, n):
    if kind == "cluster":
        return I.cluster_workload(7 * n + 1, n=n, radius=2.0 + 0.9 * n ** (1.0 / 3.0))
    pots = I.serve_potentials()
    return I.serve_request(n, kind, n, 0.05, 900.0, pots)


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n", [("cluster", 1), ("cluster", 2), ("cluster", 31), ("cluster", 33), ("Si", 513),
                                    ("Fe", 1024), ("Fe", 4900), ("Si", 32000), ("Si", 34000), ("Fe", 230000)])
def test_sets_and_lists(orc, kind, n):
    from paper_2502_19081_gb300 import mix
    wl = _workload(kind, n)
    ctx = mix.open_context(wl, precision=mix.MIX_FP32)
    for move in range(2):          # forced build, then a step
        flags, act_e, act_c = ctx.sets()
        assert np.array_equal(act_e, np.flatnonzero(flags & 4))
        assert np.array_equal(act_c, np.flatnonzero(flags & 8))
        lam, _ = ctx.lam()
        st = ctx.stats()
        assert st["n_exp"] == act_e.size and st["n_cheap"] == act_c.size
        assert st["n_core"] == int((lam == 1.0).sum()) and st["n_ramp"] == int(((lam > 0) & (lam < 1)).sum())
        nnb, nbr, rev = ctx.neighbours()
        assert st["max_neighbours"] == (int(nnb.max()) if nnb.size else 0)
        # every entry's partner lists it back at the reverse slot, rows ascending
        used = np.arange(nbr.shape[1])[None, :] < nnb[:, None]
        i, s = np.nonzero(used)
        j, r = nbr[i, s], rev[i, s]
        assert np.array_equal(nbr[j, r], i)
        assert (np.diff(nbr, axis=1)[used[:, 1:]] > 0).all()
        if n <= 5000:
            x = ctx.get_state()[0]
            assert np.array_equal(flags & 15, orc.Model(wl).sets(x) & 15)
        ctx.step(1.0, 1)
        ctx.sync()
    ctx.close()
