"""Device-built trees and lists at the sizes and forms where the builder can go
wrong (one cell, one walk chunk and a few, leaf and group sizes either way
round, coincident particles, far and tiny coordinates) against the oracle's
builder on the same positions."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hh():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1602_02832_gb300 as hh
    return hh


def _positions(form, n):
    x, v, m = synth.plummer(n, 61)
    if form == "tiny":
        x = x * 2.0 ** -90
    elif form == "huge":
        x = x * 2.0 ** 90
    elif form == "far":
        x = x + np.array([4096.0, -512.0, 7.0])
    elif form == "pairs":            # every second particle on top of its neighbour: cells down to the last level
        x[1::2] = x[: n // 2 * 2: 2]
    elif form == "clump":            # more than a leaf (and a group) at one point
        x[: n // 3] = x[0]
    elif form == "line":
        x[:, 1:] = 0.0
    return x, v, m


@pytest.mark.parametrize("form,n,leaf,n_crit,theta,order", [
    ("plummer", 2, 8, 64, 0.5, "morton"), ("plummer", 2, 1, 1, 0.5, "morton"), ("plummer", 8, 8, 64, 0.5, "morton"),
    ("plummer", 9, 8, 4, 0.5, "hilbert"), ("plummer", 33, 1, 8, 0.7, "morton"), ("plummer", 150, 8, 32, 0.5, "morton"),
    ("plummer", 2049, 32, 8, 0.6, "morton"), ("plummer", 5000, 1, 300, 0.8, "hilbert"),
    ("plummer", 4000, 8, 64, 0.0, "hilbert"), ("plummer", 4000, 8, 64, 30.0, "morton"),
    ("tiny", 3000, 8, 64, 0.5, "morton"), ("huge", 3000, 8, 64, 0.5, "hilbert"), ("far", 3000, 8, 64, 0.5, "morton"),
    ("pairs", 3001, 1, 16, 0.5, "morton"), ("clump", 900, 8, 64, 0.5, "hilbert"), ("line", 3000, 4, 40, 0.6, "morton"),
    ("plummer", 120000, 8, 256, 0.75, "morton"), ("plummer", 190000, 1, 512, 1.2, "morton")])
def test_device_tree_forms(hh, orc, form, n, leaf, n_crit, theta, order):
    x, v, m = _positions(form, n)
    z = np.zeros_like(x)
    T = orc.tree_build(x, v, z, z, m, leaf=leaf, n_crit=n_crit, theta=theta, order=order)
    cfg = hh.hh_config_default()
    cfg.theta, cfg.n_crit, cfg.leaf = theta, n_crit, leaf
    cfg.order = hh.HH_ORDER_HILBERT if order == "hilbert" else hh.HH_ORDER_MORTON
    with hh.Context(cfg, n, n + T.n_cells, 2 * len(T.list_idx) + 1024, T.n_groups + 8) as ctx:  # (cells just fit)
        ctx.hh_load_particles(x.T, v.T, m)
        ctx.hh_set_rebuild_device(True)
        for _ in range(2):           # the second build starts from the first one's order
            ctx.hh_rebuild(0.0)
        ids = ctx.hh_get_ids()
        off, idx, gof = ctx.hh_get_lists()
        nodes = ctx.hh_get_j(n, ctx.nj - n)
    assert np.array_equal(ids, T.perm) and np.array_equal(gof, T.group_of)
    assert len(nodes["m"]) == T.n_cells
    # sums of at most n terms of one sign, in another order: within n eps of each node's mass
    np.testing.assert_allclose(nodes["m"], T.node_m, rtol=max(4, n) * 2.3e-16)
    scale = np.abs(x).max()
    np.testing.assert_allclose(nodes["x"].T, T.node_x, rtol=0, atol=max(4, n) * 2.3e-16 * scale)
    assert len(off) - 1 == T.n_groups
    diff = sum(1 for g in range(T.n_groups)
               if not np.array_equal(idx[off[g]:off[g + 1]], T.list_idx[T.list_off[g]:T.list_off[g + 1]]))
    assert diff <= T.n_groups // 1000, diff   # (a tie of an opening test at its last bit)


def test_batched_rebuild_grows_some_lists(hh):
    # contexts of a batch whose lists do not fit take the entries again; the
    # others keep theirs: all equal a build alone with room enough
    sizes, ctxs, alone = (700, 3000, 1500, 3000), [], []
    cfg = hh.hh_config_default()
    cfg.precision = hh.HH_MIXED
    for k, n in enumerate(sizes):
        x, v, m = synth.plummer(n, 70 + k)
        for lst, room in ((ctxs, 16 if k % 2 else 400 * n), (alone, 400 * n)):
            c = hh.Context(cfg, n, 3 * n, room, n)
            c.hh_load_particles(x.T, v.T, m)
            c.hh_set_rebuild_device(True)
            lst.append(c)
    with hh.Batch(hh.HH_MIXED, max_sims=len(sizes), max_steps=8) as b:
        assert b.hh_batch_rebuild(ctxs, 0.0) == [hh.HH_OK] * len(sizes)
    for c, d in zip(ctxs, alone):
        d.hh_rebuild(0.0)
        assert c.nj == d.nj and all(np.array_equal(p, q) for p, q in zip(c.hh_get_lists(), d.hh_get_lists()))
        act = np.arange(c.n, dtype=np.int32)
        for e in (c, d):
            e.hh_predict(0.0)
        assert all(np.array_equal(p, q) for p, q in zip(c.hh_force(act), d.hh_force(act)))
        c.close()
        d.close()
