"""Workloads of libhh through its public entry points, for timing and for comparing outputs.

The cases are the calls that a program using this library makes, over the range of sizes that the repository's tests
and benchmark run (N = 10^3 clusters to N = 2^18 and beyond, both forms, lists from a tree or all-pairs lists):

  eval      hh_predict + hh_force / hh_force_dev on lists that the program brings itself (hh_set_j, hh_set_lists);
  static    hh_force_static on the caller's own device tensors;
  interval  one tree interval of block steps (hh_batch_run, one simulation) from a stored state, read back afterwards;
  ensemble  the same for many clusters of uneven size in shared launches;
  run       hh_load_particles + hh_run over two tree intervals + read-back (the library's own tree loop);
  snapshot  hh_load_particles + hh_rebuild on the device + forces of every particle;
  rebuild   hh_batch_rebuild of many clusters (tree, groups, lists, node records).

Inputs are Plummer spheres in standard units (M = G = -4E = 1), equal or Salpeter masses.  The lists of `eval` and
`static` come from a small octree written here, so that their exact answers need none of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DEV = "cuda"
EPS2 = 1e-8
DT_TREE = 2.0 ** -6

# tile shapes that the autotuner finds for single simulations
TUNED = {"fp64": dict(n_crit=64, tile_i=8, tile_j=256, work_item=2048, work_split=2048, tile_j_small=64),
         "mixed": dict(n_crit=128, tile_i=32, tile_j=512, work_item=8192, work_split=513, tile_j_small=128)}


def listed():
    return [
        # a small block step of a program with its own integrator: a few due particles, results to the host
        dict(name="block24-fp64-16384", kind="eval", form="fp64", n=16384, act=24, theta=0.5, n_crit=64, salpeter=False,
             host=True),
        # one force evaluation of a small cluster (the benchmark's N = 4096 configuration): tree lists, all-pairs lists
        dict(name="eval-fp64-4096", kind="eval", form="fp64", n=4096, act=4096, theta=0.5, n_crit=64, salpeter=False,
             host=False),
        dict(name="direct-mixed-4096", kind="eval", form="mixed", n=4096, act=4096, theta=0.0, n_crit=64,
             salpeter=False, host=False),
        # every particle of the benchmark's cluster in full precision: start-up forces and energy checks
        dict(name="eval-fp64-65536", kind="eval", form="fp64", n=65536, act=65536, theta=0.5, n_crit=64,
             salpeter=False, host=False),
        # a large block step of a large cluster with a mass spectrum: a quarter of the particles, odd sizes
        dict(name="eval-mixed-200003", kind="eval", form="mixed", n=200003, act=50001, theta=0.5, n_crit=128,
             salpeter=True, host=False),
        # a program that cannot allocate device memory
        dict(name="static-fp64-12007", kind="static", form="fp64", n=12007, act=3001, theta=0.5, n_crit=64,
             salpeter=False),
        # the benchmark's loop (N = 65536, tuned shapes), one interval, in both forms
        dict(name="interval-fp64-65536", kind="interval", form="fp64", n=65536, salpeter=False),
        dict(name="interval-mixed-65536", kind="interval", form="mixed", n=65536, salpeter=False),
        # many independent clusters (N log-uniform, three opening angles) advanced in shared launches
        dict(name="ensemble-mixed-24", kind="ensemble", form="mixed", count=24, n_lo=1024, n_hi=32768),
        # the shortest program: load, run, read back
        dict(name="run-mixed-8192", kind="run", form="mixed", n=8192, salpeter=False),
        # forces of a given snapshot: load, build the tree on the GPU, evaluate every particle
        dict(name="snapshot-mixed-262144", kind="snapshot", form="mixed", n=262144, salpeter=True),
        # the rebuilds of a batch of clusters at the end of an interval
        dict(name="rebuild-32", kind="rebuild", form="mixed", count=32, n_lo=1024, n_hi=32768),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "static", "interval", "ensemble", "run", "snapshot", "rebuild"])
    form = rng.choice(["fp64", "mixed"])
    salpeter = rng.random() < 0.5
    if kind == "eval":
        n = _log_int(rng, 1024, 50000 if form == "fp64" else 200000)
        act = n if rng.random() < 0.4 else _log_int(rng, 1, n)
        theta = 0.0 if n <= 4096 and rng.random() < 0.2 else round(rng.uniform(0.4, 0.75), 3)
        return dict(kind=kind, form=form, n=n, act=act, theta=theta, n_crit=rng.choice([32, 64, 100, 128, 256]),
                    salpeter=salpeter, host=act <= 512 and rng.random() < 0.5)
    if kind == "static":
        n = _log_int(rng, 512, 30000)
        return dict(kind=kind, form=form, n=n, act=_log_int(rng, 1, min(n, 6000)),
                    theta=round(rng.uniform(0.4, 0.75), 3), n_crit=rng.choice([32, 48, 64, 128]), salpeter=salpeter)
    if kind in ("ensemble", "rebuild"):
        lo = _log_int(rng, 1024, 4096)
        return dict(kind=kind, form="mixed", count=rng.randint(2, 24), n_lo=lo, n_hi=_log_int(rng, 2 * lo, 32768))
    n = _log_int(rng, 1024, {"interval": 60000, "run": 12000, "snapshot": 250000 if form == "mixed" else 40000}[kind])
    return dict(kind=kind, form=form, n=n, salpeter=salpeter)


# ------------------------------------------------------------------ inputs
def _plummer(n, rng, salpeter):
    """Positions and velocities [3, n] and masses [n] of a Plummer sphere in standard units."""
    def directions():
        c = rng.uniform(-1.0, 1.0, n)
        f = rng.uniform(0.0, 2.0 * math.pi, n)
        s = np.sqrt(1.0 - c * c)
        return np.stack([s * np.cos(f), s * np.sin(f), c])

    r = 1.0 / np.sqrt(rng.uniform(1e-9, 0.999, n) ** (-2.0 / 3.0) - 1.0)
    q = np.empty(0)
    while q.size < n:  # speed fractions with density ~ q^2 (1 - q^2)^(7/2), by rejection
        u, y = rng.uniform(0.0, 1.0, 4 * n + 64), rng.uniform(0.0, 0.1, 4 * n + 64)
        q = np.concatenate([q, u[y < u * u * (1.0 - u * u) ** 3.5]])
    x = r * directions() * (3.0 * math.pi / 16.0)
    v = q[:n] * math.sqrt(2.0) * (1.0 + r * r) ** -0.25 * directions() * math.sqrt(16.0 / (3.0 * math.pi))
    m = np.full(n, 1.0 / n)
    if salpeter:  # dN/dm ~ m^-2.35 over a factor of 100
        p = -1.35
        m = (1.0 + rng.uniform(0.0, 1.0, n) * (100.0 ** p - 1.0)) ** (1.0 / p)
        m /= m.sum()
    return x - (m * x).sum(1)[:, None], v - (m * v).sum(1)[:, None], m


def _spread_bits(k):
    out = torch.zeros_like(k)
    for b in range(21):
        out |= ((k >> b) & 1) << (3 * b)
    return out


def _tree_lists(x, theta, n_crit, leaf=8):
    """Octree over the points x [3, n] (numpy): the order of the particles, the cells (begin, end in that order), and
    per group of at most n_crit particles its list (particle p as p, cell c as n + c), ascending: off, idx, group_of."""
    n = x.shape[1]
    X = torch.tensor(x, device=DEV)
    lo = X.amin(1, keepdim=True)
    side0 = float((X - lo).max()) * (1.0 + 1e-12)
    grid = ((X - lo) * (2.0 ** 21 / side0)).long().clamp_(0, 2 ** 21 - 1)
    key = (_spread_bits(grid[0]) << 2) | (_spread_bits(grid[1]) << 1) | _spread_bits(grid[2])
    key, order = torch.sort(key, stable=True)
    X = X[:, order]
    begin, end, level, parent, first = [], [], [], [], 0  # cells, level by level
    b, e, pa = (torch.tensor([v], device=DEV) for v in (0, n, -1))
    for lv in range(22):
        begin.append(b), end.append(e), parent.append(pa), level.append(torch.full_like(b, lv))
        split = ((e - b) > leaf) if lv < 21 else torch.zeros_like(b, dtype=torch.bool)
        if not bool(split.any()):
            break
        pre = key >> (3 * (20 - lv))
        cut = torch.ones(n, dtype=torch.bool, device=DEV)
        cut[1:] = pre[1:] != pre[:-1]
        s = cut.nonzero()[:, 0]
        t = torch.cat([s[1:], torch.tensor([n], device=DEV)])
        own = torch.searchsorted(b, s, right=True) - 1
        ok = (own >= 0) & (s < e[own.clamp(min=0)]) & split[own.clamp(min=0)]
        pa = own[ok] + first
        first += b.numel()
        b, e = s[ok], t[ok]
    begin, end, level, parent = (torch.cat(u) for u in (begin, end, level, parent))
    count, cells = end - begin, begin.numel()
    kids = torch.zeros(cells, dtype=torch.long, device=DEV)
    kids.scatter_add_(0, parent[1:], torch.ones(cells - 1, dtype=torch.long, device=DEV))
    kid0 = torch.searchsorted(parent, torch.arange(cells, device=DEV))  # parents ascend, so children lie together
    up = count[parent.clamp(min=0)]
    up[0] = n_crit + 1
    group = ((count <= n_crit) & (up > n_crit)).nonzero()[:, 0]
    group = group[torch.argsort(begin[group])]
    g_of = torch.repeat_interleave(torch.arange(group.numel(), device=DEV), count[group])
    box = [torch.full((3, group.numel()), w, dtype=torch.float64, device=DEV).scatter_reduce(
        1, g_of.expand(3, n), X, how) for w, how in ((math.inf, "amin"), (-math.inf, "amax"))]
    # centres of the cells by mass are the caller's; the opening test here takes the centres of the members' positions
    C = np.concatenate([np.zeros((3, 1)), np.cumsum(X.cpu().numpy(), axis=1)], axis=1)
    hb, he = begin.cpu().numpy(), end.cpu().numpy()
    com = torch.tensor((C[:, he] - C[:, hb]) / (he - hb), device=DEV)
    size = side0 * 2.0 ** -level.double()
    g = torch.arange(group.numel(), device=DEV)
    c = torch.zeros_like(g)
    lists = []  # (group, entry)

    def members(g, c):
        k = count[c]
        at = torch.arange(int(k.sum()), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
        lists.append((torch.repeat_interleave(g, k), torch.repeat_interleave(begin[c], k) + at))

    while g.numel():
        gap = torch.maximum(torch.maximum(box[0][:, g] - com[:, c], com[:, c] - box[1][:, g]), torch.zeros((), device=DEV))
        holds = (begin[c] <= begin[group[g]]) & (end[c] >= end[group[g]])
        far = ~holds & (size[c] < theta * gap.square().sum(0).sqrt()) & (count[c] > 1)
        lists.append((g[far], n + c[far]))
        flat = ~far & ((kids[c] == 0) | (c == group[g]))
        members(g[flat], c[flat])
        deep = ~far & ~flat
        g, c = g[deep], c[deep]
        k = kids[c]
        at = torch.arange(int(k.sum()), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
        g, c = torch.repeat_interleave(g, k), torch.repeat_interleave(kid0[c], k) + at
    gi, ei = (torch.cat(u) for u in zip(*lists))
    both = torch.sort(gi * (1 << 32) + ei)[0]
    off = torch.zeros(group.numel() + 1, dtype=torch.long, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(both >> 32, minlength=group.numel()), 0)
    idx = (both & 0xFFFFFFFF).int()
    return order.cpu().numpy(), hb, he, off, idx, g_of.int()


def _list_problem(case, seed):
    """j entries (particles in tree order, then the cells as particles), lists, and the active particles."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    x, v, m = _plummer(n, rng, case["salpeter"])
    order, cb, ce, off, idx, g_of = _tree_lists(x, case["theta"], case["n_crit"])
    x, v, m = x[:, order], v[:, order], m[order]
    # accelerations and jerks of the smooth sphere; block times up to t
    s = (x * x).sum(0) + (3.0 * math.pi / 16.0) ** 2
    a = -x * s ** -1.5
    jk = -v * s ** -1.5 + 3.0 * (x * v).sum(0) * x * s ** -2.5
    t = 3.0 * 2.0 ** -9
    dt = 2.0 ** -rng.integers(7, 14, n).astype(np.float64)
    tj = np.floor(t / dt) * dt
    cum = lambda u: np.concatenate([[0.0], np.cumsum(m * u)])  # noqa: E731
    cm = cum(np.ones(n))
    cm = cm[ce] - cm[cb]
    node = [np.stack([(c[ce] - c[cb]) / cm for c in map(cum, u)]) for u in (x, v, a, jk)]
    J = [np.ascontiguousarray(np.concatenate([u, w], axis=1)) for u, w in zip((x, v, a, jk), node)]
    act = np.sort(rng.choice(n, case["act"], replace=False)).astype(np.int32)
    return dict(n=n, J=J, m=np.concatenate([m, cm]), tj=np.concatenate([tj, np.zeros(len(cm))]), t=t, off=off, idx=idx,
                g_of=g_of, act=act)


def _config(hh, form, **over):
    c = hh.hh_config_default()
    c.eps2, c.eta, c.eta_s = EPS2, 0.02, 0.01
    c.dt_tree = c.dt_max = DT_TREE
    c.precision = hh.HH_FP64 if form == "fp64" else hh.HH_MIXED
    for k, w in over.items():
        setattr(c, k, w)
    return c


def _context(hh, cfg, n):
    """Room for a tree of n particles (lists grow on the device)."""
    return hh.Context(cfg, n, 2 * n + 64, 64 * n + 4096, n // 2 + 64)


def _advance(batch, ctxs, t_end):
    while True:
        _, tn, _ = batch.hh_batch_run(ctxs, t_end)
        if (tn > t_end).all():
            return


class _Stored:
    """A simulation's synchronised state, lists and steps at the start of a tree interval."""

    def __init__(self, hh, cfg, n, rng, salpeter):
        x, v, m = _plummer(n, rng, salpeter)
        self.ctx = _context(hh, cfg, n)
        self.ctx.hh_load_particles(x, v, m)
        self.ctx.hh_set_rebuild_device(True)
        self.ctx.hh_run(0.0, 0.0)

    def store(self):
        j = self.ctx.hh_get_j(0, self.ctx.nj)
        self.j = [torch.tensor(j[k], device=DEV) for k in ("x", "v", "a", "jk", "m", "t")]
        self.dt = self.ctx.hh_get_state()["dt"]

    def restore(self):
        self.ctx.hh_set_j_dev(0, *self.j)
        self.ctx.hh_set_dt(self.dt)


def _clusters(case):
    """(size, opening angle) of each cluster: sizes spread over the logarithm, angles in turn."""
    lo, hi, k = math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"]
    return [(int(round(math.exp(lo + (hi - lo) * (q + 0.5) / k))), (0.3, 0.5, 0.7)[q % 3]) for q in range(k)]


def prepare(case, seed):
    import paper_1602_02832_gb300 as hh

    kind = case["kind"]
    st = dict(kind=kind, hh=hh)
    if kind in ("eval", "static"):
        p = _list_problem(case, seed)
        nj, k = len(p["m"]), case["act"]
        st.update(t=p["t"], act=p["act"], act_dev=torch.tensor(p["act"], device=DEV), host=case.get("host", False),
                  out=[torch.zeros(s, dtype=torch.float64, device=DEV) for s in ((3, k), (3, k), (k,))])
        if kind == "static":
            x, v = _predicted(p)
            st.update(args=(x, v, torch.tensor(p["m"], device=DEV), p["off"], p["idx"], st["act_dev"],
                            p["g_of"][st["act_dev"].long()].contiguous(), *st["out"]),
                      precision=hh.HH_FP64 if case["form"] == "fp64" else hh.HH_MIXED)
            return st
        off, idx = p["off"].cpu().numpy(), p["idx"].cpu().numpy()
        ctx = hh.Context(_config(hh, case["form"], n_crit=case["n_crit"]), p["n"], nj, len(idx), len(off) - 1)
        ctx.hh_set_j(0, *p["J"], p["m"], p["tj"])
        ctx.hh_set_lists(p["n"], nj, off, idx, p["g_of"].cpu().numpy())
        st.update(ctx=ctx)
        return st
    rng = np.random.default_rng(seed)
    if kind in ("run", "snapshot"):
        x, v, m = _plummer(case["n"], rng, case["salpeter"])
        ctx = _context(hh, _config(hh, case["form"]), case["n"])
        ctx.hh_set_rebuild_device(True)
        st.update(ctx=ctx, xvm=(x, v, m))
        if kind == "snapshot":
            n = case["n"]
            st.update(act_dev=torch.arange(n, dtype=torch.int32, device=DEV),
                      out=[torch.zeros(s, dtype=torch.float64, device=DEV) for s in ((3, n), (3, n), (n,))])
        return st
    if kind == "interval":
        sims = [_Stored(hh, _config(hh, case["form"], **TUNED[case["form"]]), case["n"], rng, case["salpeter"])]
    else:
        sims = [_Stored(hh, _config(hh, case["form"], theta=theta, n_crit=64, work_item=8192), n, rng, False)
                for n, theta in _clusters(case)]
    batch = hh.Batch(sims[0].ctx.cfg.precision, max_sims=len(sims), max_steps=4096)
    ctxs = [s.ctx for s in sims]
    _advance(batch, ctxs, DT_TREE)
    batch.hh_batch_rebuild(ctxs, DT_TREE)
    for s in sims:
        s.store()
    st.update(sims=sims, ctxs=ctxs, batch=batch)
    return st


# -------------------------------------------------------------------- one pass
def run(st):
    kind = st["kind"]
    if kind == "static":
        st["hh"].hh_force_static(*st["args"], eps2=EPS2, precision=st["precision"])
        return st["out"]
    if kind == "eval":
        ctx = st["ctx"]
        ctx.hh_predict(st["t"])
        if st["host"]:
            return list(ctx.hh_force(st["act"]))
        ctx.hh_force_dev(st["act_dev"], *st["out"])
        return st["out"]
    if kind == "run":
        ctx = st["ctx"]
        ctx.hh_load_particles(*st["xvm"])
        ctx.hh_run(0.0, 2 * DT_TREE)
        return dict(ctx.hh_get_state(), ids=ctx.hh_get_ids())
    if kind == "snapshot":
        ctx = st["ctx"]
        ctx.hh_load_particles(*st["xvm"])
        ctx.hh_rebuild(0.0)
        ctx.hh_predict(0.0)
        ctx.hh_force_dev(st["act_dev"], *st["out"])
        return st["out"] + [ctx.hh_get_ids()]
    if kind == "rebuild":
        # (the state stays at this time: a rebuild can be taken again)
        st["batch"].hh_batch_rebuild(st["ctxs"], DT_TREE)
        return [c.hh_get_ids() for c in st["ctxs"]]
    for s in st["sims"]:
        s.restore()
    _advance(st["batch"], st["ctxs"], 2 * DT_TREE)
    if kind == "interval":
        return st["ctxs"][0].hh_get_state()
    # up to 64 outputs: every cluster's state as one array
    return [np.concatenate([u.ravel() for u in c.hh_get_state().values()]) for c in st["ctxs"]]


# ------------------------------------------------------------------- the work
def work(case):
    """Bytes: state in, results out, and each list index once; flops: 60 per pair term.  Pair counts follow the mean
    list length of a Plummer sphere, about 120 log2(n) - 300 entries at theta 0.5 and n_crit 64 (n entries at
    theta 0), growing as theta^-2, and the block steps of an interval take about 8 steps per particle."""
    kind = case["kind"]

    def mean_list(n, theta=0.5):
        if theta == 0.0:
            return float(n)
        return min(float(n), max(100.0, 120.0 * math.log2(n) - 300.0) * (0.5 / max(theta, 0.05)) ** 2)

    if kind in ("eval", "static"):
        n, k, ln = case["n"], case["act"], mean_list(case["n"], case["theta"])
        groups = min(k, max(1.0, n / (0.28 * case["n_crit"])))
        return {"bytes": 1.4 * n * 112 + groups * ln * 4 + k * 60, "flops": 60.0 * k * ln}
    if kind in ("ensemble", "rebuild"):
        n = (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])  # mean of a log-uniform size
        sims = case["count"]
    else:
        n, sims = case["n"], 1
    lists = 4.0 * mean_list(n) * n / 18.0
    if kind in ("snapshot", "rebuild"):
        force = kind == "snapshot"
        return {"bytes": sims * (n * 56 + 1.4 * n * 112 + lists + n * 56 * force + n * 8),
                "flops": sims * n * (60.0 * mean_list(n) * force + 100.0)}
    steps = {"interval": 8.0, "ensemble": 8.0, "run": 20.0}[kind]
    return {"bytes": sims * (1.4 * n * 112 * 2 + lists), "flops": sims * 60.0 * steps * n * mean_list(n)}


# -------------------------------------------------------------- exact answers
def _predicted(p):
    x, v, a, jk = (torch.tensor(u, device=DEV) for u in p["J"])
    d = p["t"] - torch.tensor(p["tj"], device=DEV)
    return x + d * (v + d / 2 * (a + d / 3 * jk)), v + d * (a + d / 2 * jk)


def exact(case, seed):
    """The list sums in 64 bits for the cases whose lists are made here; the others integrate or build trees."""
    if case["kind"] not in ("eval", "static"):
        return None
    p = _list_problem(case, seed)
    x, v = _predicted(p)
    m, off, idx = torch.tensor(p["m"], device=DEV), p["off"], p["idx"].long()
    act = torch.tensor(p["act"], device=DEV).long()
    g = p["g_of"][act].long()
    length = off[g + 1] - off[g]
    out = torch.zeros((7, len(act)), dtype=torch.float64, device=DEV)
    done = torch.cumsum(length, 0)
    at = 0
    while at < len(act):  # about 2^22 pairs at a time
        base = int(done[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(done, base + (1 << 22), right=True)))
        ln = length[at:to]
        slot = torch.repeat_interleave(torch.arange(to - at, device=DEV), ln)
        e = torch.arange(int(ln.sum()), device=DEV) - torch.repeat_interleave(torch.cumsum(ln, 0) - ln, ln)
        j, i = idx[off[g[at:to]][slot] + e], act[at:to][slot]
        dx, dv = x[:, j] - x[:, i], v[:, j] - v[:, i]
        r2 = (dx * dx).sum(0) + EPS2
        mj = torch.where(j == i, 0.0, m[j])
        u = mj / (r2 * r2.sqrt())
        terms = torch.cat([u * dx, u * (dv - 3.0 * (dx * dv).sum(0) / r2 * dx), (-mj / r2.sqrt())[None]])
        out[:, at:to].index_add_(1, slot, terms)
        at = to
    return [out[:3].contiguous(), out[3:6].contiguous(), out[6].contiguous()]
