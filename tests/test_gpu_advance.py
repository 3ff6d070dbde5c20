"""hh_advance's persistent loop against its graph loop (taken with per-launch timing on), bit for bit.

Shapes with and without work items, runs cut into several launches, a state that breaks the block rule (left to the
graph loop, counters included), and contexts advanced by several threads at once."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

KEYS = ("x", "v", "a", "jk", "t", "dt")


@pytest.fixture(scope="module")
def hh():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1602_02832_gb300 as hh
    return hh


def _ctx(hh, prec, n, seed=1, **over):
    x, v, m = synth.plummer_salpeter(n, seed)
    c = hh.hh_config_default()
    c.precision = hh.HH_FP64 if prec == "fp64" else hh.HH_MIXED
    for k, val in over.items():
        setattr(c, k, val)
    ctx = hh.Context(c, n, 2 * n + 64, 64 * n * max(1, n // 16) + 4096, n)
    ctx.hh_load_particles(x.T, v.T, m)
    ctx.hh_run(0.0, 0.0)
    return ctx


def _both(ctxs, t_end):
    """Advances the first context in the persistent loop, the second in the graph loop; states and counters agree."""
    ctxs[1].hh_force_timing(1)
    steps = [c.hh_advance(t_end) for c in ctxs]
    assert steps[0] == steps[1]
    s0, s1 = (c.hh_get_state() for c in ctxs)
    for k in KEYS:
        assert np.array_equal(s0[k], s1[k]), k
    c0, c1 = (c.hh_get_counters() for c in ctxs)
    assert c0 == c1
    assert np.array_equal(ctxs[0].hh_get_tile_histogram(), ctxs[1].hh_get_tile_histogram())
    return steps[0]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,over", [(2, {}), (300, {}), (1500, dict(work_item=2048)), (5000, dict(tile_i=8, n_crit=48)),
                                    (3000, dict(work_item=2048, work_split=64, tile_j_small=64))])
def test_persistent_equals_graph(hh, prec, n, over):
    ctxs = [_ctx(hh, prec, n, **over) for _ in range(2)]
    _both(ctxs, 0.0)  # nothing due yet
    assert _both(ctxs, 2.0 ** -6) > 0
    for c in ctxs:
        c.hh_rebuild(2.0 ** -6)
    assert _both(ctxs, 2.0 ** -5) > 0


def test_several_launches(hh):
    ctxs = [_ctx(hh, "mixed", 2000) for _ in range(2)]
    assert _both(ctxs, 8 * 2.0 ** -6) > 600  # more than two launches of 256 steps


@pytest.mark.parametrize("broken", ["time", "overdue"])
def test_state_off_the_block_rule(hh, broken):
    ctxs = [_ctx(hh, "fp64", 600) for _ in range(2)]
    for c in ctxs:
        s = c.hh_get_state()
        m = c.hh_get_j(0, c.n)["m"]
        dt = np.full(c.n, 2.0 ** -9)
        t = np.full(c.n, 2.0 ** -8)
        if broken == "time":
            t += 0.3 * 2.0 ** -9  # no multiple of the step
        else:
            t[5:] += 2.0 ** -7    # particles 0 to 4 are due before the others' time
        c.hh_set_j(0, s["x"], s["v"], s["a"], s["jk"], m, t)
        c.hh_set_dt(dt)
        c.hh_reset_counters()
    assert _both(ctxs, 2.0 ** -6) > 0


def test_contexts_in_threads(hh):
    specs = [("mixed", 900, 3), ("fp64", 700, 4), ("mixed", 4000, 5), ("fp64", 2500, 6)]
    alone = []
    for prec, n, seed in specs:
        c = _ctx(hh, prec, n, seed)
        c.hh_advance(2.0 ** -6)
        alone.append(c.hh_get_state())
    ctxs = [_ctx(hh, *s) for s in specs]
    err = []

    def go(c):
        try:
            c.hh_advance(2.0 ** -6)
        except Exception as e:  # noqa: BLE001
            err.append(e)

    th = [threading.Thread(target=go, args=(c,)) for c in ctxs]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not err
    for c, s in zip(ctxs, alone):
        got = c.hh_get_state()
        for k in KEYS:
            assert np.array_equal(got[k], s[k]), k
