"""hh_advance while a batch launch that leaves SMs free runs in another thread:
it takes free SMs instead of waiting for the launch to end."""
import threading
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("left", [8, 32])
def test_advance_on_the_sms_a_batch_leaves(left):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1602_02832_gb300 as hh

    def ctx(n, seed):
        x, v, m = synth.plummer(n, seed)
        cfg = hh.hh_config_default()
        c = hh.Context(cfg, n, 2 * n + 64, 64 * n + 4096, n)
        c.hh_set_rebuild_device(True)
        c.hh_load_particles(x.T, v.T, m)
        c.hh_run(0.0, 0.0)
        return c

    alone = ctx(1024, 32)
    alone.hh_advance(2.0 ** -9)
    big, small = ctx(60000, 31), ctx(1024, 32)
    with hh.Batch(hh.HH_FP64, max_sims=1, max_steps=4096) as b:
        b.hh_batch_set_ctas(-left)
        started, done = threading.Event(), threading.Event()

        def go():
            started.set()
            b.hh_batch_run([big], [2.0 ** -6])  # some 50 ms
            done.set()

        th = threading.Thread(target=go)
        th.start()
        started.wait()
        time.sleep(0.004)  # the launch is on the GPU
        small.hh_advance(2.0 ** -9)  # some 1 ms
        beside = not done.is_set()
        th.join()
    assert beside
    s0, s1 = alone.hh_get_state(), small.hh_get_state()
    assert all(np.array_equal(s0[k], s1[k]) for k in s0)
    for c in (alone, big, small):
        c.close()
