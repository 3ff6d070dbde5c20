"""hh_advance with step limits beyond the persistent loop's levels (2^-31 to 1):
steps that start inside them and leave them on the way, against the graph loop
(taken with per-launch timing on), bit for bit, counters included."""
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


def _ctx(hh, prec, x, v, m, dt, **over):
    n = len(m)
    c = hh.hh_config_default()
    c.precision = hh.HH_FP64 if prec == "fp64" else hh.HH_MIXED
    for k, val in over.items():
        setattr(c, k, val)
    ctx = hh.Context(c, n, 3 * n + 64, n * n + 4096, n)
    ctx.hh_load_particles(x.T, v.T, m)
    ctx.hh_run(0.0, 0.0)
    steps = np.empty(n)
    steps[:] = dt[ctx.hh_get_ids()]
    ctx.hh_set_dt(steps)
    ctx.hh_reset_counters()
    return ctx


def _both(hh, t_end, *args, **over):
    ctxs = [_ctx(hh, *args, **over) for _ in range(2)]
    ctxs[1].hh_force_timing(1)
    steps = [c.hh_advance(t_end) for c in ctxs]
    assert steps[0] == steps[1] == ctxs[0].hh_get_counters()["block_steps"]
    s0, s1 = (c.hh_get_state() for c in ctxs)
    for k in s0:
        assert np.array_equal(s0[k], s1[k]), k
    assert ctxs[0].hh_get_counters() == ctxs[1].hh_get_counters()
    assert np.array_equal(ctxs[0].hh_get_tile_histogram(), ctxs[1].hh_get_tile_histogram())
    assert (s0["t"] + s0["dt"] > t_end).all()
    for c in ctxs:
        c.close()
    return steps[0], s0["dt"]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_steps_below_the_levels(hh, prec):
    # a pair 2e-7 apart among 62 others: its steps begin at 2^-31 and shrink to 2^-35 and below
    x, v, m = (u.copy() for u in synth.plummer(64, 11))
    x[1] = x[0] + np.array([2e-7, 0.0, 0.0])
    v[1] = v[0] + np.array([0.0, 0.9 * np.sqrt(2 * m[0] / 2e-7), 0.0])
    dt = np.full(64, 2.0 ** -20)
    dt[:2] = 2.0 ** -31
    steps, got = _both(hh, 2.0 ** -25, prec, x, v, m, dt, dt_min=2.0 ** -40, eps2=0.0)
    assert steps > 300 and got.min() < 2.0 ** -31


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_steps_above_the_levels(hh, prec):
    # a wide soft cluster: steps begin at 1/4 and double to more than 1
    x, v, m = synth.plummer(300, 12)
    steps, got = _both(hh, 64.0, prec, 60.0 * x, v / 8.0, m, np.full(300, 0.25), dt_tree=64.0, dt_max=64.0, eps2=4.0)
    assert steps > 20 and got.max() > 1.0


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_batched_run_refuses_steps_outside_the_levels(hh, prec):
    x, v, m = (u.copy() for u in synth.plummer(64, 11))
    x[1] = x[0] + np.array([2e-7, 0.0, 0.0])
    v[1] = v[0] + np.array([0.0, 0.9 * np.sqrt(2 * m[0] / 2e-7), 0.0])
    dt = np.full(64, 2.0 ** -20)
    dt[:2] = 2.0 ** -31
    c = _ctx(hh, prec, x, v, m, dt, dt_min=2.0 ** -40, eps2=0.0)
    new = _ctx(hh, prec, x, v, m, dt, dt_min=2.0 ** -40, eps2=0.0)
    lists = c.hh_get_lists()
    with hh.Batch(c.cfg.precision, max_sims=1, max_steps=64) as b:
        with pytest.raises(hh.HHError) as e:
            b.hh_batch_run([c], [2.0 ** -25])
        assert e.value.code == hh.HH_EINVAL
    assert all(np.array_equal(p, q) for p, q in zip(lists, c.hh_get_lists()))
    y, u, k = synth.plummer(64, 13)
    for q in (c, new):  # loaded again, the context is as good as another
        q.hh_load_particles(y.T, u.T, k)
        q.hh_run(0.0, 2.0 ** -6)
    s0, s1 = c.hh_get_state(), new.hh_get_state()
    assert all(np.array_equal(s0[f], s1[f]) for f in s0)
    c.close()
    new.close()
