"""Thin systems in the plain form's force kernel: every component as good as FP64 sums of its own terms.

Sheets whose separations (and velocities) have one component far below the others, alone, in a list with a few entries
off the sheet, and with every component zero; active counts around the kernel's warps and slices."""
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
    """acc, jerk of the particles act, all with the one list idx."""
    dev = torch.device("cuda", 0)
    t = lambda u, dt: torch.tensor(np.ascontiguousarray(u), dtype=dt, device=dev)  # noqa: E731
    k = len(act)
    out = [torch.zeros(s, dtype=torch.float64, device=dev) for s in ((3, k), (3, k), (k,))]
    hh.hh_force_static(t(x, torch.float64), t(v, torch.float64), t(m, torch.float64), t([0, len(idx)], torch.int64),
                       t(idx, torch.int32), t(act, torch.int32), t(np.zeros(k), torch.int32), *out, eps2=eps2,
                       precision=hh.HH_FP64)
    return np.concatenate([out[0].cpu().numpy(), out[1].cpu().numpy()])


def _reference(x, v, m, idx, act, eps2):
    """Sums [6, k] in long double from the FP64 differences' exact values, and the sums of each component's own sizes."""
    x, v, m = (np.asarray(u, dtype=np.longdouble) for u in (x, v, m))
    ref, size = [], []
    for i in act:
        j = idx[idx != i]
        d, w = x[:, j] - x[:, [i]], v[:, j] - v[:, [i]]
        r2 = (d * d).sum(0) + np.longdouble(eps2)
        u = m[j] / (r2 * np.sqrt(r2))
        q = u * 3 * ((d * w).sum(0) / r2)
        ref.append(np.concatenate([(u * d).sum(1), (u * w - q * d).sum(1)]))
        size.append(np.concatenate([np.abs(u * d).sum(1), (np.abs(u * w) + np.abs(q * d)).sum(1)]))
    return np.array(ref).T, np.array(size).T


@pytest.mark.parametrize("axis", [0, 2])
@pytest.mark.parametrize("places", [4, 12, 24, 40])
@pytest.mark.parametrize("k", [1, 3, 17, 32])
@pytest.mark.parametrize("n_list", [60, 700, 5000])
def test_sheets(env, axis, places, k, n_list):
    hh, torch = env
    rng = np.random.default_rng([axis, places, k, n_list])
    n = n_list + 40
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.exp(rng.uniform(-4, 4, n)) / n
    x[axis] *= 2.0 ** -places
    v[axis] *= 2.0 ** -places
    idx, act = np.sort(rng.choice(n, n_list, replace=False)), np.sort(rng.choice(n, k, replace=False))
    got = _static(hh, torch, x, v, m, idx, act, 1e-8)
    ref, size = _reference(x, v, m, idx, act, 1e-8)
    # FP64 sums in any order (at most 2048 terms a thread and part), or the integers where they are better
    assert (np.abs(got - ref) <= 2.0 ** -41 * size).all()


@pytest.mark.parametrize("k", [1, 17, 32])
def test_one_particle_off_the_sheet(env, k):
    # its own forces are round, the others' are not: the tile is judged particle by particle
    hh, torch = env
    rng = np.random.default_rng(k)
    n = 900
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.full(n, 1.0 / n)
    x[2] *= 1e-9
    v[2] *= 1e-9
    act = np.arange(k)
    x[2, 0], v[2, 0] = 0.7, -0.4
    idx = np.arange(k, n)
    got = _static(hh, torch, x, v, m, idx, act, 1e-8)
    ref, size = _reference(x, v, m, idx, act, 1e-8)
    assert (np.abs(got - ref) <= 2.0 ** -41 * size).all()


def test_motion_in_a_plane(env):
    hh, torch = env
    rng = np.random.default_rng(9)
    n = 3000
    x, v, m = rng.normal(size=(3, n)), rng.normal(size=(3, n)), np.full(n, 1.0 / n)
    x[1] = 0.25
    v[1] = 0.0
    act, idx = np.arange(0, n, 100), np.arange(n)
    got = _static(hh, torch, x, v, m, idx, act, 1e-8)
    ref, size = _reference(x, v, m, idx, act, 1e-8)
    assert not got[1].any() and not got[4].any()
    assert (np.abs(got - ref) <= 2.0 ** -41 * size).all()
