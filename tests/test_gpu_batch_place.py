"""Results of a simulation in a batch and its place there: beyond the first 256
simulations (whose block times a CTA keeps in shared memory) a step takes the
same list parts as before them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hh():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1602_02832_gb300 as hh
    return hh


def _listed(hh, prec, n, nj, n_list, group, seed, own=True, **over):
    """n particles among nj entries, a random list of n_list entries per group of `group` (own: the group's particles
    among them), all due at 2^-7."""
    rng = np.random.default_rng(seed)
    cfg = hh.hh_config_default()
    cfg.precision = prec
    for k, val in over.items():
        setattr(cfg, k, val)
    groups = (n + group - 1) // group
    c = hh.Context(cfg, n, nj, groups * n_list, groups)
    x = rng.normal(size=(3, nj))
    z = np.zeros((3, nj))
    c.hh_set_j(0, x, 0.1 * rng.normal(size=(3, nj)), z, z, np.full(nj, 1.0 / nj), np.zeros(nj))
    idx = rng.integers(n if nj > n else 0, nj, (groups, n_list))
    if own:
        idx[:, :group] = np.arange(groups)[:, None] * group + np.arange(group)
    idx = np.sort(idx, axis=1).astype(np.int32).ravel()
    c.hh_set_lists(n, nj, np.arange(groups + 1) * n_list, idx, (np.arange(n) // group).astype(np.int32))
    c.hh_set_dt(np.full(n, 2.0 ** -7))
    return c


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("own", [True, False])
def test_a_list_mode_step_at_any_place(hh, prec, own):
    # 512 due particles with lists of 200 entries among 2^18: predicted from the lists alone (2^18 > 512 * 200 * 2)
    # where the step's data are kept in shared memory, entry by entry where they are not
    P = hh.HH_FP64 if prec == "fp64" else hh.HH_MIXED
    over = dict(tile_i=8, tile_j=256, work_item=2048, work_split=2048, tile_j_small=64)
    small = [_listed(hh, P, 2, 2, 2, 2, s, **over) for s in range(256)]
    states = []
    with hh.Batch(P, max_sims=257, max_steps=8) as b:
        for first in (True, False):
            big = _listed(hh, P, 512, 1 << 18, 200, 8, 999, own, **over)
            sims = [big] + small if first else small + [big]
            _, tn, _ = b.hh_batch_run(sims, [2.0 ** -7] * 257, max_steps=1)
            assert big.hh_get_counters()["list_steps"] == (1 if first else 0)
            states.append(big.hh_get_state())
            big.close()
    for k in states[0]:
        assert np.array_equal(states[0][k], states[1][k]), k
    for c in small:
        c.close()


def test_an_advance_of_many_particles_predicts_every_entry(hh):
    # 2^22 particles due at once: hh_advance does not take list steps, however many are due
    n = 1 << 22
    cfg = hh.hh_config_default()
    with hh.Context(cfg, n, n, n // 16, n // 32) as c:
        x = np.stack([np.arange(n) % 2048.0, np.arange(n) // 2048.0, np.zeros(n)])
        z = np.zeros((3, n))
        c.hh_set_j(0, x, z, z, z, np.full(n, 1.0 / n), np.zeros(n))
        idx = (np.arange(n // 32)[:, None] * 32 + np.arange(2)).astype(np.int32).ravel()
        c.hh_set_lists(n, n, np.arange(n // 32 + 1) * 2, idx, (np.arange(n) // 32).astype(np.int32))
        c.hh_set_dt(np.full(n, 2.0 ** -7))
        assert c.hh_advance(2.0 ** -7) == 1
        k = c.hh_get_counters()
    assert k["particle_steps"] == n and k["list_steps"] == 0
