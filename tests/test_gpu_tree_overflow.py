"""A device build whose cells do not fit: refused before it reads or writes
anything of the tree that was there, alone and inside a batch, and the context
goes on with a build that fits."""
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


def _ctx(hh, n_max, cells, groups, prec):
    cfg = hh.hh_config_default()
    cfg.precision = prec
    c = hh.Context(cfg, n_max, n_max + cells, 400 * n_max, groups)
    c.hh_set_rebuild_device(True)
    return c


def _snap(c):
    return dict(c.hh_get_j(0, c.nj), ids=c.hh_get_ids(), **{f"l{q}": u for q, u in enumerate(c.hh_get_lists())})


def _same(a, b):
    assert a.keys() == b.keys()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


# groups_max below and above the refused tree's groups; no cell at all to a few too few
@pytest.mark.parametrize("groups", [100, 400])
@pytest.mark.parametrize("cells", [1, 700, 1500])
@pytest.mark.parametrize("batched", [False, True])
def test_refused_build_leaves_the_context_as_it_was(hh, cells, groups, batched):
    small, big, last = synth.plummer(60, 1), synth.plummer(4000, 2), synth.plummer_salpeter(61, 3)
    for prec in (hh.HH_FP64, hh.HH_MIXED):
        c, other = _ctx(hh, 4000, cells, groups, prec), _ctx(hh, 4000, 8000, 4000, prec)
        with hh.Batch(prec, max_sims=2, max_steps=8) as b:

            def rebuild(data, ok):
                c.hh_load_particles(data[0].T, data[1].T, data[2])
                other.hh_load_particles(big[0].T, big[1].T, big[2])
                if batched:
                    rcs = b.hh_batch_rebuild([other, c], 0.0, check=False)
                    assert rcs == [hh.HH_OK, hh.HH_OK if ok else hh.HH_ENOMEM]
                elif ok:
                    c.hh_rebuild(0.0)
                else:
                    with pytest.raises(hh.HHError) as e:
                        c.hh_rebuild(0.0)
                    assert e.value.code == hh.HH_ENOMEM and "nj_max" in str(e.value)

            if cells > 1:
                rebuild(small, True)  # another tree's cells and groups in the builder's buffers
            for _ in range(2):
                rebuild(big, False)
                s = c.hh_get_state()
                assert np.array_equal(s["x"], big[0].T) and np.array_equal(s["v"], big[1].T)
                assert np.array_equal(c.hh_get_ids(), np.arange(4000))
                with pytest.raises(hh.HHError) as e:
                    c.hh_step()
                assert e.value.code == hh.HH_ESTATE
            if cells > 1:
                rebuild(last, True)
                new = _ctx(hh, 4000, 8000, 4000, prec)
                new.hh_load_particles(last[0].T, last[1].T, last[2])
                new.hh_rebuild(0.0)
                _same(_snap(c), _snap(new))
                new.close()
            if batched:
                alone = _ctx(hh, 4000, 8000, 4000, prec)
                alone.hh_load_particles(big[0].T, big[1].T, big[2])
                alone.hh_rebuild(0.0)
                _same(_snap(other), _snap(alone))
                alone.close()
        c.close()
        other.close()
