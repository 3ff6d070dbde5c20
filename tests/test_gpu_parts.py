"""Large evaluations of the plain form take longer list parts than small ones
of the same particles: the pair terms are the same, only the order of the sums
differs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile_j", [(6000, 128), (20000, 128), (20000, 512)])
def test_all_at_once_equals_a_few_at_a_time(n, tile_j):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1602_02832_gb300 as hh
    x, v, m = synth.plummer(n, 81)
    cfg = hh.hh_config_default()
    cfg.n_crit, cfg.theta, cfg.tile_j = 16, 0.5, tile_j
    with hh.Context(cfg, n, 3 * n, 64 * n, n) as c:
        c.hh_load_particles(x.T, v.T, m)
        c.hh_set_rebuild_device(True)
        c.hh_rebuild(0.0)
        c.hh_predict(0.0)
        acc, jerk, pot = c.hh_force(np.arange(n, dtype=np.int32))
        off, idx, gof = c.hh_get_lists()
        J = c.hh_get_j(0, c.nj)
        some = np.linspace(0, n - 1, 41).astype(np.int32)
        a2, j2, p2 = c.hh_force(some)
    for q, p in enumerate(some):
        e = idx[off[gof[p]]:off[gof[p] + 1]]
        e = e[e != p]
        d, w = J["x"][:, e] - J["x"][:, [p]], J["v"][:, e] - J["v"][:, [p]]
        r = np.sqrt((d * d).sum(0) + cfg.eps2)
        # the sum of each of at most 128 slices and of each part is rounded, and so is each addition of
        # them: fewer than 2 (128 + parts) roundings of at most the sum of the terms' sizes, on both sides
        tol = 4 * (128 + len(e) / 128 + 2) * 2.0 ** -53
        assert np.abs(acc[:, p] - a2[:, q]).max() <= tol * (J["m"][e] / r ** 2).sum()
        assert np.abs(jerk[:, p] - j2[:, q]).max() <= tol * (4 * J["m"][e] * np.sqrt((w * w).sum(0)) / r ** 3).sum()
        assert abs(pot[p] - p2[q]) <= tol * (J["m"][e] / r).sum()
