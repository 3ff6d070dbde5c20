"""The plain form's force kernel at the edges of its integer pair term, through hh_force_static.

List lengths and active counts around the kernel's chunks, slices and parts; softenings from none to dominant; lists
with entries that the integers leave to FP64 (their part is summed again in FP64), infinities and NaN among them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    import paper_1602_02832_gb300 as hh
    return hh, torch


def _static(hh, torch, x, v, m, idx, act, eps2):
    """acc, jerk, pot of the particles act, all with the one list idx."""
    dev = torch.device("cuda", 0)
    t = lambda u, dt: torch.tensor(np.ascontiguousarray(u), dtype=dt, device=dev)  # noqa: E731
    k = len(act)
    out = [torch.zeros(s, dtype=torch.float64, device=dev) for s in ((3, k), (3, k), (k,))]
    hh.hh_force_static(t(x, torch.float64), t(v, torch.float64), t(m, torch.float64), t([0, len(idx)], torch.int64),
                       t(idx, torch.int32), t(act, torch.int32), t(np.zeros(k), torch.int32), *out, eps2=eps2,
                       precision=hh.HH_FP64)
    return np.concatenate([out[0].cpu().numpy(), out[1].cpu().numpy(), out[2].cpu().numpy()[None]])


def _reference(x, v, m, idx, act, eps2, dtype):
    """Sums [7, k] and sums of the terms' sizes, self skipped."""
    x, v, m = (np.asarray(u, dtype=dtype) for u in (x, v, m))
    ref, size = [], []
    for i in act:
        j = idx[idx != i]
        d, w = x[:, j] - x[:, [i]], v[:, j] - v[:, [i]]
        with np.errstate(all="ignore"):
            r2 = (d * d).sum(0) + dtype(eps2)
            p = m[j] / np.sqrt(r2)
            u = p / r2
            ref.append(np.concatenate([(u * d).sum(1), (u * (w - 3 * ((d * w).sum(0) / r2) * d)).sum(1), [-p.sum()]]))
            a, b = (np.abs(u) * np.sqrt((q * q).sum(0)) for q in (d, w))
            size.append([a.sum()] * 3 + [b.sum()] * 3 + [np.abs(p).sum()])
    return np.array(ref).T, np.array(size).T


@pytest.mark.parametrize("n_list", [1, 2, 127, 128, 129, 255, 257, 2047, 2048, 2049, 5000])
@pytest.mark.parametrize("k", [1, 3, 9, 31, 32, 33])
def test_edges_of_chunks_and_slices(env, n_list, k):
    hh, torch = env
    rng = np.random.default_rng(n_list * 100 + k)
    n = max(n_list, k) + 5
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.exp(rng.uniform(-4, 4, n)) / n
    idx = np.sort(rng.choice(n, n_list, replace=False))
    act = np.sort(rng.choice(n, k, replace=False))
    for eps2 in (0.0, 1e-8, 0.3, 1e4):
        got = _static(hh, torch, x, v, m, idx, act, eps2)
        ref, size = _reference(x, v, m, idx, act, eps2, np.longdouble)
        # per term: the differences' rounding (2^-53 each, at most 5 of them in a term) and 2^-51; then at most 128
        # slice partials and a few parts are added in FP64 (a tree of about 12 levels): 2^-48 of the sizes in all
        assert (np.abs(got - ref) <= 2.0 ** -48 * size).all()


@pytest.mark.parametrize("what", ["zero mass", "negative mass", "large mass", "far", "fast", "coincident"])
def test_parts_left_to_fp64(env, what):
    hh, torch = env
    rng = np.random.default_rng(5)
    n, eps2 = 4500, 1e-8
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.full(n, 1.0 / n)
    at = 2500  # in the second of three parts
    if what == "zero mass":
        m[at] = 0.0
    elif what == "negative mass":
        m[at] = -0.25
    elif what == "large mass":
        m[at] = 1e70
    elif what == "far":
        x[0, at] = 1e70
    elif what == "fast":
        v[1, at] = 1e70
    else:
        x[:, at], eps2 = x[:, 7], 0.0
    idx, act = np.arange(n), np.array([0, 7, 100, 101, 4499])
    got = _static(hh, torch, x, v, m, idx, act, eps2)
    ref, size = _reference(x, v, m, idx, act, eps2, np.float64)
    fine = np.isfinite(ref)
    assert fine[:, 0].all() and fine.all() == (what != "coincident")
    # FP64 sums in another order: at most 2048 terms a thread and part, 2^-41 of the sizes
    assert (np.abs(got - ref)[fine] <= 2.0 ** -41 * size[fine]).all()
    assert np.array_equal(np.isnan(ref), np.isnan(got)) and np.array_equal(np.isinf(ref), np.isinf(got))


@pytest.mark.parametrize("n_act,n_list", [(4000, 250), (4000, 700), (4000, 1500), (8000, 2000), (8192, 2048)])
def test_static_part_lengths(env, n_act, n_list):
    # every active particle is a tile of its own (two lists in turn): at most 8192 parts of at most 2048 entries
    hh, torch = env
    rng = np.random.default_rng(n_act + n_list)
    n, eps2 = 2 * n_list + 11, 1e-4
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.full(n, 1.0 / n)
    lists = [np.sort(rng.choice(n, n_list, replace=False)) for _ in range(2)]
    act, gid = rng.integers(0, n, n_act), np.arange(n_act) % 2
    dev = torch.device("cuda", 0)
    t = lambda u, dt: torch.tensor(np.ascontiguousarray(u), dtype=dt, device=dev)  # noqa: E731
    out = [torch.zeros(s, dtype=torch.float64, device=dev) for s in ((3, n_act), (3, n_act), (n_act,))]
    hh.hh_force_static(t(x, torch.float64), t(v, torch.float64), t(m, torch.float64),
                       t([0, n_list, 2 * n_list], torch.int64), t(np.concatenate(lists), torch.int32),
                       t(act, torch.int32), t(gid, torch.int32), *out, eps2=eps2, precision=hh.HH_FP64)
    got = np.concatenate([out[0].cpu().numpy(), out[1].cpu().numpy(), out[2].cpu().numpy()[None]])
    for g in range(2):
        sel = np.flatnonzero(gid == g)[:: max(1, n_act // 400)]
        ref, size = _reference(x, v, m, lists[g], act[sel], eps2, np.float64)
        assert (np.abs(got[:, sel] - ref) <= 2.0 ** -41 * size).all()
