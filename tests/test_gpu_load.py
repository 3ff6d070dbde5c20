"""Loading particles into a context that has built its tree on the device: the
checks run on the device, a refused load leaves everything as it was, and an
accepted one gives what a new context gives."""
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


def _ctx(hh, prec, n_max):
    cfg = hh.hh_config_default()
    cfg.precision = prec
    c = hh.Context(cfg, n_max, 3 * n_max, 400 * n_max, n_max)
    c.hh_set_rebuild_device(True)
    return c


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_second_load_equals_a_new_context(hh, prec):
    P = hh.HH_FP64 if prec == "fp64" else hh.HH_MIXED
    used, new = _ctx(hh, P, 3000), _ctx(hh, P, 3000)
    x, v, m = synth.plummer(3000, 5)
    used.hh_load_particles(x.T, v.T, m)
    used.hh_run(0.0, 2.0 ** -6)
    y, u, k = synth.plummer_salpeter(2001, 6)        # fewer than before
    for c in (used, new):
        c.hh_load_particles(y.T, u.T, k, 2.0 ** -6)
        assert np.array_equal(c.hh_get_ids(), np.arange(2001)) and c.nj == 2001
        j = c.hh_get_j(0, 2001)
        assert np.array_equal(j["x"], y.T) and np.array_equal(j["v"], u.T) and np.array_equal(j["m"], k)
        assert not j["a"].any() and not j["jk"].any() and (j["t"] == 2.0 ** -6).all()
        c.hh_run(2.0 ** -6, 2.0 ** -5)
    a, b = used.hh_get_state(), new.hh_get_state()
    assert all(np.array_equal(a[q], b[q]) for q in a) and np.array_equal(used.hh_get_ids(), new.hh_get_ids())
    used.close()
    new.close()


@pytest.mark.parametrize("what,q,value,word", [("x", 0, np.nan, "non-finite"), ("x", 1699, np.inf, "non-finite"),
                                               ("v", 300, -np.inf, "non-finite"), ("m", 0, 0.0, "masses"),
                                               ("m", 1699, -1.0, "masses"), ("m", 5, np.nan, "masses"),
                                               ("m", 6, np.inf, "masses"), ("t", 0, np.nan, "time")])
def test_refused_load_changes_nothing(hh, what, q, value, word):
    c = _ctx(hh, hh.HH_MIXED, 2000)
    x, v, m = synth.plummer(2000, 7)
    c.hh_load_particles(x.T, v.T, m)
    c.hh_run(0.0, 2.0 ** -6)
    before, ids, lists = c.hh_get_j(0, c.nj), c.hh_get_ids(), c.hh_get_lists()
    y, u, k = (s.copy() for s in synth.plummer(1700, 8))
    t = value if what == "t" else 0.0
    if what != "t":
        (y[q].__setitem__(2, value) if what == "x" else u[q].__setitem__(0, value) if what == "v" else k.__setitem__(q, value))
    with pytest.raises(hh.HHError) as e:
        c.hh_load_particles(y.T, u.T, k, t)
    assert e.value.code == hh.HH_EINVAL and word in str(e.value)
    after = c.hh_get_j(0, c.nj)
    assert all(np.array_equal(before[f], after[f]) for f in before) and np.array_equal(ids, c.hh_get_ids())
    assert all(np.array_equal(p, r) for p, r in zip(lists, c.hh_get_lists()))
    c.hh_advance(2.0 ** -5)                           # (and the run goes on: base records as they were)
    d = _ctx(hh, hh.HH_MIXED, 2000)
    d.hh_load_particles(x.T, v.T, m)
    d.hh_run(0.0, 2.0 ** -6)
    d.hh_advance(2.0 ** -5)
    a, b = c.hh_get_state(), d.hh_get_state()
    assert all(np.array_equal(a[f], b[f]) for f in a)
    c.close()
    d.close()


def test_ids_after_lists_of_fewer_particles(hh):
    # lists set by the caller for another number of particles start new ids,
    # also when the last ones were kept by the device builder
    c = _ctx(hh, hh.HH_FP64, 1000)
    x, v, m = synth.plummer(1000, 9)
    c.hh_load_particles(x.T, v.T, m)
    c.hh_rebuild(0.0)
    assert not np.array_equal(c.hh_get_ids(), np.arange(1000))
    z = np.zeros((3, 10))
    c.hh_set_j(0, x[:10].T, v[:10].T, z, z, m[:10], np.zeros(10))
    c.hh_set_lists(10, 10, np.array([0, 10]), np.arange(10, dtype=np.int32), np.zeros(10, np.int32))
    assert np.array_equal(c.hh_get_ids(), np.arange(10))
    c.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n_new", [1500, 900])
def test_load_leaves_the_entries_behind_its_particles(hh, prec, n_new):
    # a program's own nodes (and particles beyond the loaded ones) stay as set,
    # with and without a device builder: lists over them give the same forces
    P = hh.HH_FP64 if prec == "fp64" else hh.HH_MIXED
    x, v, m = synth.plummer(1500, 21)
    y, u, k = synth.plummer(n_new, 22)
    out = []
    for dev in (True, False):
        c = _ctx(hh, P, 1500)
        c.hh_set_rebuild_device(dev)
        c.hh_load_particles(x.T, v.T, m)
        c.hh_rebuild(0.0)
        rng = np.random.default_rng(23)
        J = [rng.normal(size=(3, 2000)) for _ in range(4)]
        mj = rng.uniform(0.5, 1.0, 2000) / 2000
        c.hh_set_j(0, *J, mj, np.zeros(2000))
        c.hh_load_particles(y.T, u.T, k)
        off = np.arange(0, 51) * 400
        idx = np.sort(rng.integers(0, 2000, (50, 400)), axis=1).astype(np.int32).ravel()
        c.hh_set_lists(1500, 2000, off, idx, (np.arange(1500) // 30).astype(np.int32))
        j = c.hh_get_j(0, 2000)
        for q, f in enumerate(("x", "v", "a", "jk")):
            assert np.array_equal(j[f][:, n_new:], J[q][:, n_new:]), (dev, f)
        assert np.array_equal(j["m"][n_new:], mj[n_new:]) and np.array_equal(j["m"][:n_new], k)
        assert np.array_equal(j["x"][:, :n_new], y.T) and not j["a"][:, :n_new].any()
        c.hh_predict(2.0 ** -10)
        out.append(c.hh_force(np.arange(1500, dtype=np.int32)))
        c.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
