"""What the framework's users have it do, at the sizes they do it: cases for timing and comparing.

A case names a kind of work, a seeded Chung-Lu graph (the recipe of ``synth.chung_lu``, drawn on
the GPU here: power-law expected degrees on both layers, distinct edges in random order, random
ids), and what is asked of it. Every call goes through the package's public entry points
(``ABCore``), on device tensors unless the case says ``host``.

kinds
  peel        one or several single (alpha, beta)-cores of a loaded graph, one call each
  pruned      the same after core numbers were prepared (Algorithm 2, GCC+)
  batch       a grid of pairs in one ``compute_batch`` call
  load        a new edge list: build both CSR layers, then one core
  cores       a new edge list: build, then every vertex's core number
  components  component labels of a loaded graph
  community   the component of a core that holds a query vertex
  serve       a serving session: start with targets, a stream of edge updates, stop
"""

import math

import numpy as np
import torch

from paper_2606_07148_gb300 import ABCore, abi

DEV = "cuda"


def _case(name, kind, nU, nV, m, gu, gv, pairs, **more):
    c = dict(kind=kind, nU=nU, nV=nV, m=m, gu=gu, gv=gv, kmax=0, pairs=pairs)
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # the smallest graph in the repository's workloads: one query, where launches and latency count
        _case("peel-20k", "peel", 2000, 1500, 20_000, 2.3, 2.3, "2:3", kmax=200),
        # five separate queries on an ordinary graph, queued without waiting (the plain single peel)
        _case("peel-80M-five", "peel", 4_000_000, 2_000_000, 80_000_000, 2.1, 2.4,
              "2:2 5:3 10:10 20:5 50:50", queued=True),
        # the billion-edge recipe at a fifth of the size: one deep query on a large graph
        _case("peel-300M", "peel", 20_000_000, 10_000_000, 300_000_000, 2.0, 2.3, "64:64"),
        # the five queries again for a user who prepared core numbers once
        _case("pruned-80M-five", "pruned", 4_000_000, 2_000_000, 80_000_000, 2.1, 2.4,
              "2:2 5:3 10:10 20:5 50:50"),
        # a small grid on a small graph with odd layer sizes, masks in new tensors each call
        _case("batch-200k-64", "batch", 10_007, 5_003, 200_000, 2.1, 2.2, "grid:8:1:64"),
        # the 16 x 16 grid on an ordinary graph, masks in buffers the caller keeps
        _case("batch-100M-256", "batch", 4_000_000, 2_000_000, 100_000_000, 2.1, 2.2, "grid:16:1:512",
              kept=True),
        # a small edge list from numpy to numpy: load, one core, masks on the host
        _case("load-200k-host", "load", 10_007, 5_003, 200_000, 2.1, 2.2, "5:5", host=True),
        # a large edge list on the device: load, one core
        _case("load-80M", "load", 4_000_000, 2_000_000, 80_000_000, 2.1, 2.4, "10:10"),
        # preprocessing of the pruned query on a new graph with odd layer sizes
        _case("cores-20M", "cores", 999_983, 500_009, 20_000_000, 2.1, 2.4, ""),
        # component labels of the ordinary graph
        _case("components-80M", "components", 4_000_000, 2_000_000, 80_000_000, 2.1, 2.4, ""),
        # community search on a mid-size graph with odd layer sizes
        _case("community-8M", "community", 400_009, 199_999, 8_000_000, 2.1, 2.3, "5:5"),
        # a serving session of 2000 updates against the four targets of the serving workload
        _case("serve-200k", "serve", 10_000, 5_000, 200_000, 2.1, 2.2, "2:2 5:5 10:20 32:32", ops=2000),
    ]


# per kind: the range of edge counts a drawn case takes (no more than the listed largest)
_EDGES = {
    "peel": (10_000, 300_000_000),
    "pruned": (1_000_000, 80_000_000),
    "batch": (20_000, 60_000_000),
    "load": (20_000, 80_000_000),
    "cores": (100_000, 20_000_000),
    "components": (20_000, 80_000_000),
    "community": (100_000, 20_000_000),
    "serve": (20_000, 400_000),
}


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(sorted(_EDGES))
    m = logint(*_EDGES[kind])
    # average degrees as in the workloads: 10 to 25 on U, 1 to 3 times that on V
    nU = max(200, int(m / rng.uniform(10.0, 25.0)))
    nV = max(100, int(nU / rng.uniform(1.0, 3.0)))
    gu, gv = round(rng.uniform(2.0, 2.4), 2), round(rng.uniform(2.1, 2.5), 2)
    top = max(4, min(64, int(2 * math.sqrt(m) / 30)))

    def pair():
        return "%d:%d" % (logint(1, top), logint(1, top))

    c = _case("", kind, nU, nV, m, gu, gv, "")
    if kind in ("peel", "pruned"):
        c["pairs"] = " ".join(pair() for _ in range(rng.choice((1, 1, 2, 5))))
        c["queued"] = rng.random() < 0.5
        if kind == "peel":
            c["host"] = m < 10_000_000 and rng.random() < 0.25
    elif kind == "batch":
        c["pairs"] = "grid:%d:1:%d" % (rng.choice((4, 8, 12)), logint(16, 512))
        c["kept"] = rng.random() < 0.5
    elif kind == "load":
        c["pairs"] = pair()
        c["host"] = m < 10_000_000 and rng.random() < 0.5
        c["csr"] = bool(c["host"]) and rng.random() < 0.5
    elif kind == "community":
        c["pairs"] = pair()
    elif kind == "serve":
        c["pairs"] = " ".join(sorted({pair() for _ in range(rng.choice((1, 2, 4)))}))
        c["ops"] = 2 * rng.randrange(100, 1000)
    return c


# ---- inputs ---------------------------------------------------------------------------------

def _weights(n, gamma, m, kmax):
    """Expected degrees in rank order: a power law clipped to [1, kmax], summing to m."""
    w = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-1.0 / (gamma - 1.0))
    w *= m / w.sum()
    for _ in range(20):
        w.clamp_(1.0, kmax)
        free = (w > 1.0) & (w < kmax)
        rest, fixed = w[free].sum(), w[~free].sum()
        if rest <= 0:
            break
        w[free] *= ((m - fixed) / rest).clamp(min=0.0)
    return w


def _edges(case, seed):
    """m distinct edges in random order: int32 tensors on the device, and the generator."""
    nU, nV, m = case["nU"], case["nV"], case["m"]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 2654435761 % (1 << 31) + 17)
    kmax = float(case["kmax"] or math.isqrt(m))
    cu = torch.cumsum(_weights(nU, case["gu"], m, kmax), 0)
    cv = torch.cumsum(_weights(nV, case["gv"], m, kmax), 0)
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    while keys.numel() < m:
        k = m - keys.numel()
        k += k // 4 + 64
        u = torch.rand(k, dtype=torch.float64, device=DEV, generator=g).mul_(cu[-1])
        v = torch.rand(k, dtype=torch.float64, device=DEV, generator=g).mul_(cv[-1])
        iu = torch.searchsorted(cu, u, right=True).clamp_(max=nU - 1)
        iv = torch.searchsorted(cv, v, right=True).clamp_(max=nV - 1)
        del u, v
        new = iu.mul_(nV).add_(iv)
        del iv
        keys = torch.unique(torch.cat([keys, new]))
        del new, iu
    keys = keys[torch.randperm(keys.numel(), device=DEV, generator=g)[:m]]
    pu = torch.randperm(nU, device=DEV, generator=g).to(torch.int32)
    pv = torch.randperm(nV, device=DEV, generator=g).to(torch.int32)
    eu, ev = pu[torch.div(keys, nV, rounding_mode="floor")], pv[keys % nV]
    return eu.contiguous(), ev.contiguous(), g


def _pairs(case):
    s = case["pairs"]
    if s.startswith("grid:"):
        # a k x k log-spaced grid, strictly increasing values (the repository's grid recipe)
        _, k, lo, hi = s.split(":")
        k, lo, hi = int(k), int(lo), int(hi)
        vals = []
        for i in range(k):
            r = int(math.floor(lo * (hi / lo) ** (i / (k - 1)) + 0.5))
            vals.append(max(r, vals[-1] + 1) if vals else r)
        return [(a, b) for a in vals for b in vals]
    return [tuple(int(x) for x in p.split(":")) for p in s.split()]


def _updates(case, eu, ev, g):
    """An update stream: 70 % inserts of absent edges with degree-proportional endpoints, 30 %
    deletes of present ones, then the same updates taken back in reverse order (so a session
    leaves the graph as it found it). Arrays op, u, v, target."""
    n, nV = case["ops"] // 2, case["nV"]
    m = case["m"]
    base = eu.to(torch.int64) * nV + ev

    def pick(k):
        return torch.randint(0, m, (k,), device=DEV, generator=g)

    ndel = max(1, min(int(n * 0.3), m // 4))
    dele = base[torch.randperm(m, device=DEV, generator=g)[:ndel]]
    ins = torch.empty(0, dtype=torch.int64, device=DEV)
    while ins.numel() < n - ndel:
        k = 2 * (n - ndel) + 64
        new = eu[pick(k)].to(torch.int64) * nV + ev[pick(k)]
        new = new[~torch.isin(new, base)]
        ins = torch.unique(torch.cat([ins, new]))
    ins = ins[torch.randperm(ins.numel(), device=DEV, generator=g)[: n - ndel]]
    key = torch.cat([ins, dele])
    op = torch.cat([torch.zeros_like(ins), torch.ones_like(dele)])
    order = torch.randperm(key.numel(), device=DEV, generator=g)
    key, op = key[order], op[order]
    key, op = torch.cat([key, key.flip(0)]), torch.cat([op, 1 - op.flip(0)])
    nt = len(_pairs(case))
    tg = torch.randint(0, nt, (key.numel(),), device=DEV, generator=g)
    return [x.cpu().numpy().astype(np.int64) for x in (op, key // nV, key % nV, tg)]


def prepare(case, seed):
    eu, ev, g = _edges(case, seed)
    s = dict(case=case, pairs=_pairs(case))
    core = s["core"] = ABCore(0)
    nU, nV, kind = case["nU"], case["nV"], case["kind"]
    if kind in ("load", "cores"):
        if case.get("csr"):
            order = torch.argsort(eu, stable=True)
            off = torch.zeros(nU + 1, dtype=torch.int64, device=DEV)
            off[1:] = torch.cumsum(torch.bincount(eu, minlength=nU), 0)
            s["off"], s["adj"] = off.cpu().numpy(), ev[order].cpu().numpy()
        elif case.get("host"):
            s["eu"], s["ev"] = eu.cpu().numpy(), ev.cpu().numpy()
        else:
            s["eu"], s["ev"] = eu, ev
    else:
        core.load_edges(nU, nV, eu, ev)
    if kind == "pruned":
        core.core_numbers()
    if kind == "batch":
        s["a"], s["b"] = [p[0] for p in s["pairs"]], [p[1] for p in s["pairs"]]
        if case.get("kept"):
            s["out"] = (torch.empty((len(s["pairs"]), nU), dtype=torch.uint8, device=DEV),
                        torch.empty((len(s["pairs"]), nV), dtype=torch.uint8, device=DEV))
    if case.get("host"):
        s["out"] = (np.empty(nU, dtype=np.uint8), np.empty(nV, dtype=np.uint8))
    if kind == "community":
        s["vertex"] = int(eu[0])  # an endpoint of a random edge: mostly a well-connected vertex
    if kind == "serve":
        op, u, v, tg = _updates(case, eu, ev, g)
        reqs = (abi.abcore_req * len(op))()
        for i in range(len(op)):
            reqs[i] = abi.abcore_req(int(op[i]), int(u[i]), int(v[i]), int(tg[i]), i)
        s["reqs"] = [(abi.abcore_req * len(reqs[i:i + 512]))(*reqs[i:i + 512]) for i in range(0, len(reqs), 512)]
        s["buf"] = np.zeros(4096, dtype=ABCore.RESP_DTYPE)
    return s


# ---- one pass -------------------------------------------------------------------------------

def _cores_of(core, s):
    out = []
    queued = bool(s["case"].get("queued"))
    for a, b in s["pairs"]:
        if s["case"].get("host"):
            mu, mv = core.compute(a, b, np.empty_like(s["out"][0]), np.empty_like(s["out"][1]))
        else:
            mu, mv = core.compute(a, b, *_new_masks(s) if queued else (), asynchronous=queued)
        out += [mu, mv]
    if queued and not s["case"].get("host"):
        core.sync()
    return out


def _new_masks(s):
    c = s["case"]
    return (torch.empty(c["nU"], dtype=torch.uint8, device=DEV), torch.empty(c["nV"], dtype=torch.uint8, device=DEV))


def run(s):
    core, case = s["core"], s["case"]
    kind = case["kind"]
    if kind in ("peel", "pruned"):
        return _cores_of(core, s)
    if kind == "batch":
        return list(core.compute_batch(s["a"], s["b"], *s.get("out", ())))
    if kind == "load":
        if case.get("csr"):
            core.load_csr(case["nU"], case["nV"], s["off"], s["adj"])
        else:
            core.load_edges(case["nU"], case["nV"], s["eu"], s["ev"])
        return _cores_of(core, s)
    if kind == "cores":
        core.load_edges(case["nU"], case["nV"], s["eu"], s["ev"])
        return list(core.core_numbers())
    if kind == "components":
        return list(core.components())
    if kind == "community":
        a, b = s["pairs"][0]
        return list(core.community(0, s["vertex"], a, b))
    # serve: a session over the loaded graph, requests submitted as the ring takes them
    core.serve_start(s["pairs"], ring_slots=1024)
    chunks, at, total, got = s["reqs"], 0, case["ops"], []
    n = 0
    while n < total:
        if at < len(chunks) and core.serve_submit(chunks[at]) is not None:
            at += 1
        part = core.serve_poll_into(s["buf"])
        if len(part):
            got.append(part.copy())
            n += len(part)
    core.serve_stop()
    r = np.concatenate(got)
    return [r["tag"].astype(np.int64), r["status"].astype(np.int32), r["in_core"], r["u_in"], r["v_in"]]


# ---- what a pass cannot do without ------------------------------------------------------------

def work(case):
    """Bytes of one pass: the edges once (4 bytes each from a loaded graph's adjacency, 8 as a
    list), what is built once (both layers' adjacency), and every output once. Integer work only."""
    n, m, kind = case["nU"] + case["nV"], case["m"], case["kind"]
    k = len(_pairs(case)) if case["pairs"] else 1
    if kind in ("peel", "pruned", "batch"):
        b = 4 * m + k * n
    elif kind == "load":
        b = 8 * m + 8 * m + n
    elif kind == "cores":
        b = 8 * m + 8 * m + 4 * n
    elif kind == "components":
        b = 4 * m + 4 * n
    elif kind == "community":
        b = 4 * m + n
    else:  # serve: the targets' cores once, then the requests and their answers
        b = 4 * m + 16 * case["ops"]
    return {"bytes": float(b), "flops": 0.0}


# ---- plain results ----------------------------------------------------------------------------

def _peel(eu, ev, nU, nV, a, b, mu=None, mv=None):
    """Masks (bool) of the (a, b)-core by rounds of plain counting in 64 bits."""
    mu = torch.ones(nU, dtype=torch.bool, device=DEV) if mu is None else mu.clone()
    mv = torch.ones(nV, dtype=torch.bool, device=DEV) if mv is None else mv.clone()
    live = mu[eu] & mv[ev]
    if not bool(live.all()):
        eu, ev = eu[live], ev[live]
    while True:
        du, dv = torch.bincount(eu, minlength=nU), torch.bincount(ev, minlength=nV)
        ku, kv = mu & (du >= a), mv & (dv >= b)
        same = bool((ku == mu).all()) and bool((kv == mv).all())
        mu, mv = ku, kv
        if same:
            return mu, mv
        live = mu[eu] & mv[ev]
        eu, ev = eu[live], ev[live]


def _labels(eu, ev, nU, nV):
    """Smallest unified id of each vertex's component, by repeated minima over the edges."""
    lab = torch.arange(nU + nV, dtype=torch.int64, device=DEV)
    x, y = eu, ev + nU
    while True:
        lo = torch.minimum(lab[x], lab[y])
        new = lab.scatter_reduce(0, x, lo, "amin").scatter_reduce(0, y, lo, "amin")
        new = torch.minimum(new, new[new])
        if bool((new == lab).all()):
            return lab
        lab = new


def exact(case, seed):
    kind, m, nU, nV = case["kind"], case["m"], case["nU"], case["nV"]
    pairs = _pairs(case) if case["pairs"] else []
    if m * max(1, len(pairs)) > 600_000_000:
        return None
    eu32, ev32, g = _edges(case, seed)
    eu, ev = eu32.to(torch.int64), ev32.to(torch.int64)
    if kind in ("peel", "pruned", "load"):
        out = []
        for a, b in pairs:
            out += [x.to(torch.uint8) for x in _peel(eu, ev, nU, nV, a, b)]
        return out
    if kind == "batch":
        ms = [_peel(eu, ev, nU, nV, a, b) for a, b in pairs]
        return [torch.stack([x[0] for x in ms]).to(torch.uint8), torch.stack([x[1] for x in ms]).to(torch.uint8)]
    if kind == "cores":
        cu = torch.zeros(nU, dtype=torch.int32, device=DEV)
        cv = torch.zeros(nV, dtype=torch.int32, device=DEV)
        mu = mv = None
        k = 0
        while eu.numel():
            k += 1
            mu, mv = _peel(eu, ev, nU, nV, k, k, mu, mv)
            cu[mu], cv[mv] = k, k
            live = mu[eu] & mv[ev]
            eu, ev = eu[live], ev[live]
        return [cu, cv, int(max(int(cu.max()), int(cv.max())))]
    if kind == "components":
        lab = _labels(eu, ev, nU, nV)
        return [lab[:nU].to(torch.int32), lab[nU:].to(torch.int32), int(torch.unique(lab).numel())]
    if kind == "community":
        a, b = pairs[0]
        mu, mv = _peel(eu, ev, nU, nV, a, b)
        live = mu[eu] & mv[ev]
        lab = _labels(eu[live], ev[live], nU, nV)
        q = int(eu32[0])
        in_u = mu & (lab[:nU] == lab[q]) & mu[q]
        in_v = mv & (lab[nU:] == lab[q]) & mu[q]
        return [in_u.to(torch.uint8), in_v.to(torch.uint8), int(in_u.sum() + in_v.sum())]
    if m * case["ops"] > 450_000_000:
        return None
    op, u, v, tg = _updates(case, eu32, ev32, g)
    n = len(op)
    half = n // 2
    # every updated edge is touched once in the first half: one slot each after the base edges
    ux = torch.from_numpy(u[:half]).to(DEV)
    vx = torch.from_numpy(v[:half]).to(DEV)
    alu, alv = torch.cat([eu, ux]), torch.cat([ev, vx])
    on = torch.ones(m + half, dtype=torch.bool, device=DEV)
    on[m:] = torch.from_numpy(op[:half]).to(DEV) == 1  # a deleted edge is present until then
    key = ux * nV + vx
    on[:m] = ~torch.isin(eu * nV + ev, key)            # (its base slot stands for it no longer)
    res = np.zeros((3, n), dtype=np.uint8)
    for k in range(n):
        slot = m + (k if k < half else n - 1 - k)
        on[slot] = bool(op[k] == 0)
        a, b = pairs[int(tg[k])]
        mu, mv = _peel(alu[on], alv[on], nU, nV, a, b)
        iu, iv = bool(mu[int(u[k])]), bool(mv[int(v[k])])
        res[:, k] = (iu and iv, iu, iv)
    return [np.arange(n, dtype=np.int64), np.zeros(n, dtype=np.int32), res[0], res[1], res[2]]
