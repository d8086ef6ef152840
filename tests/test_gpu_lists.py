"""Neighbour lists built a cell at a time, where that form has its edges: cell grids
beyond the 8,192 cells whose counts every CTA sums itself, stencils with more
candidates than a tile holds, empty cells, cells of one atom, box sides that are open.
Rows are integers: equal to the oracle's, entry by entry."""
import numpy as np
import pytest

from paper_2502_19081_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _gas(kind, rng):
    """positions, box, periodic, list radius, capacity"""
    if kind == "cells_12167":      # 23^3 cells of some two atoms, many empty
        L = np.full(3, 23.3 * 4.0)
        return rng.random((22000, 3)) * L, L, (1, 1, 1), 4.0, 64
    if kind == "open_z":
        L = np.array([12.5 * 4.0, 12.9 * 4.0, 8.5 * 4.0])
        return rng.random((9000, 3)) * L, L, (1, 1, 0), 4.0, 64
    # a slab of 45 atoms a cell (1,215 candidates a stencil) beside a thin gas
    L = np.array([10.2, 11.7, 10.9]) * 4.0
    a = rng.random((18000, 3)) * L * np.array([1.0, 1.0, 0.333])
    b = rng.random((2500, 3)) * L
    return np.concatenate([a, b]), L, (1, 1, 1), 4.0, 256


def _same_rows(nnb, nbr, ref):
    rn, rb = ref
    assert np.array_equal(nnb, rn)
    used = np.arange(nbr.shape[1])[None, :] < nnb[:, None]
    m = min(nbr.shape[1], rb.shape[1])
    assert not used[:, m:].any()
    assert np.array_equal(np.where(used, nbr, -1)[:, :m], np.where(used[:, :m], rb[:, :m], -1))


def _reverse_ok(nnb, nbr, rev):
    i, s = np.nonzero(np.arange(nbr.shape[1])[None, :] < nnb[:, None])
    assert np.array_equal(nbr[nbr[i, s], rev[i, s]], i)


@pytest.mark.parametrize("kind", ["cells_12167", "open_z", "dense_slab"])
def test_lists_alone(orc, kind):
    import torch
    from paper_2502_19081_gb300 import mix
    pos, L, per, rl, cap = _gas(kind, np.random.default_rng(len(kind)))
    n = len(pos)
    x = np.zeros((n, 4))
    x[:, :3] = pos
    nnb = torch.zeros(n, dtype=torch.int32, device="cuda")
    nbr = torch.zeros((n, cap), dtype=torch.int32, device="cuda")
    rev = torch.zeros((n, cap), dtype=torch.int32, device="cuda")
    st = mix.neighbours_noalloc(torch.from_numpy(x).cuda(), np.zeros(3), L, per, rl, cap, nnb, nbr, rev)
    assert st == mix.MIX_OK
    nnb, nbr, rev = nnb.cpu().numpy(), nbr.cpu().numpy(), rev.cpu().numpy()
    _same_rows(nnb, nbr, orc.neighbours(x, np.zeros(3), L, per, rl, cap))
    _reverse_ok(nnb, nbr, rev)


def test_lists_rebuilt_in_a_step(orc):
    """85,183 atoms in 10,648 cells: the rows of the step that rebuilds are the oracle's
    at the positions it rebuilt for."""
    from paper_2502_19081_gb300 import mix
    wl = I.serve_request(9, "Si", 85184, 0.01, 1500.0, I.serve_potentials())
    c = mix.open_context(wl, precision=mix.MIX_FP32)
    assert int(np.prod(c.cells()[0])) > 8192
    before = c.stats()["rebuilds"]
    for _ in range(60):
        c.step(1.0, 1)
        if c.stats()["rebuilds"] > before:
            break
    else:
        raise AssertionError("no rebuild")
    nnb, nbr, rev = c.neighbours()
    x = c.get_state()[0]
    s = wl.system
    _same_rows(nnb, nbr, orc.neighbours(x, s.box_lo, s.box_len, s.periodic,
                                        max(wl.ace.r_cut, wl.spline.r_cut) + wl.skin, c.cap))
    _reverse_ok(nnb, nbr, rev)
    c.close()
