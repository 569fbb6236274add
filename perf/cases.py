"""The work that users of mslice have it do, as cases that can be timed.

Every case goes through the package's public entry points.  Inputs are
synthetic temporal graphs of the shapes the repository's benchmark and tests
use, generated on the GPU from the seed alone:

* "planted": 4 equal blocks, p_out = p_in / 10, 10% of the nodes switch block
  over the sequence, 5% edge churn between snapshots;
* "powerlaw": degree-corrected blocks, power-law degrees (cutoff
  sqrt(n * mean degree)) and community sizes (exponent 1.5 on [20, 5000]), 5%
  edge churn;
* "contact": few people, very many snapshots with a handful of contacts each,
  drawn from a fixed pool of pairs.

The listed cases:

* solve_small     a latency-bound solve of a small graph on a kept handle (a
                  program that re-solves with other parameters)
* solve_small_new the same size from host arrays, handle and all: the first
                  thing a user runs
* solve_t16       the plain benchmark shape T = 16, n = 100,000, kept handle
* solve_t64       the long benchmark shape T = 64, built from device arrays and
                  solved once: the largest case
* solve_random    randomised refinement (theta = 1/100)
* solve_cpm_cat   the Constant Potts Model under categorical coupling, ragged n
* solve_global    the global null model, planted blocks, warm-started from
                  given labels (what a serving window solves)
* contact_long    7,375 snapshots of 327 people, from host arrays
* windows         the windowed optimisation of a contact sequence
* sweep_batch     a gamma x omega sweep of several graphs in one batch
* serve           a serving session: live graphs, snapshots submitted at once
* score           Q of a known labelling of a graph that arrives in pinned host
                  memory (build + modularity)
"""
import math

import numpy as np
import torch

import paper_2608_03695_gb300 as mslice

CHURN = 0.05


class Snapshot:
    """Symmetric CSR of one snapshot (arrays or tensors)."""

    def __init__(self, indptr, indices, weights):
        self.indptr, self.indices, self.weights = indptr, indices, weights

    def host(self, pin=False):
        if pin:
            return Snapshot(*(x.cpu().pin_memory() for x in (self.indptr, self.indices, self.weights)))
        return Snapshot(*(x.cpu().numpy() for x in (self.indptr, self.indices, self.weights)))


# --------------------------------------------------------------------------
# inputs


def _csr(s, u, v, n, T, w_max, salt):
    """Snapshots from edge lists (s: snapshot of every edge; repeats and
    self-loops are dropped).  The weight is a hash of the pair, so an edge
    keeps it over the sequence."""
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    keep = a != b
    key = torch.unique((s[keep] * n + a[keep]) * n + b[keep])
    b = key % n
    row = torch.div(key, n, rounding_mode="floor")
    s = torch.div(row, n, rounding_mode="floor")
    a = row - s * n
    key = torch.cat([key, (s * n + b) * n + a])
    del row, s, a, b
    key = torch.sort(key).values
    col = key % n
    row = torch.div(key, n, rounding_mode="floor")
    lo, hi = torch.minimum(row % n, col), torch.maximum(row % n, col)
    h = (lo * 2654435761 + hi * 40503 + salt * 97) & 0x7FFFFFFF
    h = (h ^ (h >> 13)) * 1274126177 & 0x7FFFFFFF
    w = ((h ^ (h >> 11)) % w_max + 1).to(torch.int32)
    deg = torch.bincount(row, minlength=n * T)
    ptr = torch.zeros(n * T + 1, dtype=torch.int64, device=key.device)
    torch.cumsum(deg, 0, out=ptr[1:])
    first = ptr[: n * T].view(T, n)
    ends = ptr[n::n].view(T, 1)
    indptr = torch.cat([first, ends], 1) - first[:, :1]
    cut = [0] + ptr[n::n].tolist()
    col = col.to(torch.int32)
    return [Snapshot(indptr[t], col[cut[t]:cut[t + 1]], w[cut[t]:cut[t + 1]]) for t in range(T)]


def _churned(gen, m, T, dev):
    """m edge slots over T snapshots; a slot is drawn anew with probability
    CHURN at every step.  Returns the draw every (slot, snapshot) uses, its
    snapshot, and the number of draws."""
    new = torch.rand(m, T, generator=gen, device=dev) < CHURN
    new[:, 0] = True
    draw = torch.cumsum(new.view(-1), 0) - 1
    snap = torch.arange(T, device=dev).repeat(m)
    return draw, snap, int(draw[-1]) + 1


def _planted(n, T, mean_deg, w_max, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    blocks = 4
    block = torch.randint(0, blocks, (n,), generator=gen, device=dev)
    # the nodes that switch do so at a snapshot of their own
    when = torch.randint(1, max(T, 2), (n,), generator=gen, device=dev)
    moves = torch.rand(n, generator=gen, device=dev) < 0.1
    later = torch.where(moves, (block + 1) % blocks, block)
    draw, snap, k = _churned(gen, max(1, int(n * mean_deg / 2)), T, dev)
    u = torch.randint(0, n, (k,), generator=gen, device=dev)
    inside = torch.rand(k, generator=gen, device=dev) < 0.25 / (0.25 + 0.075)
    order = torch.argsort(block, stable=True)
    count = torch.bincount(block, minlength=blocks)
    start = torch.cumsum(count, 0) - count
    r = torch.rand(k, generator=gen, device=dev, dtype=torch.float64)
    anyone = (r * n).long().clamp(max=n - 1)
    mate_of = lambda blk: order[(start[blk] + (r * count[blk]).long().clamp(max=n)).clamp(max=n - 1)]  # noqa: E731
    v0 = torch.where(inside, mate_of(block[u]), anyone)
    v1 = torch.where(inside, mate_of(later[u]), anyone)
    uu = u[draw]
    vv = torch.where(snap >= when[uu], v1[draw], v0[draw])
    return _csr(snap, uu, vv, n, T, w_max, seed % 1000003), block.to(torch.int32)


def _powerlaw_quantile(u, exponent, lo, hi):
    a = 1.0 - exponent
    return (lo ** a + u * (hi ** a - lo ** a)) ** (1.0 / a)


def _powerlaw_mean(exponent, lo, hi):
    a1, a2 = 2.0 - exponent, 1.0 - exponent
    return (a2 / a1) * (hi ** a1 - lo ** a1) / (hi ** a2 - lo ** a2)


def _powerlaw(n, T, mean_deg, deg_exp, mixing, w_max, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    hi = math.sqrt(n * mean_deg)
    a, b = 1e-3, mean_deg
    for _ in range(80):
        mid = 0.5 * (a + b)
        a, b = (mid, b) if _powerlaw_mean(deg_exp, mid, hi) < mean_deg else (a, mid)
    theta = _powerlaw_quantile(rng.random(n), deg_exp, 0.5 * (a + b), hi)
    sizes = np.minimum(np.floor(_powerlaw_quantile(rng.random(n // 20 + 1), 1.5, 20.0, 5001.0)), 5000).astype(np.int64)
    sizes = sizes[: int(np.searchsorted(np.cumsum(sizes), n)) + 1]
    comm = np.repeat(np.arange(len(sizes)), sizes)[:n]
    comm = np.concatenate([comm, np.full(n - len(comm), len(sizes) - 1)])
    # nodes sorted by community are 0..n-1 under `order`
    order = rng.permutation(n)
    cdf = np.cumsum(theta)  # theta of the sorted nodes
    c_lo = np.searchsorted(comm, np.arange(len(sizes)), side="left")
    c_hi = np.searchsorted(comm, np.arange(len(sizes)), side="right")
    base = np.where(c_lo > 0, cdf[np.maximum(c_lo, 1) - 1], 0.0)
    mass = np.where(c_hi > c_lo, cdf[np.maximum(c_hi, 1) - 1] - base, 0.0)
    to = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
    order_d, cdf_d, comm_d, base_d, mass_d = to(order), to(cdf), to(comm.astype(np.int64)), to(base), to(mass)
    draw, snap, k = _churned(gen, max(1, int(n * mean_deg / 2)), T, dev)
    pick = lambda x: torch.searchsorted(cdf_d, x, right=True).clamp(max=n - 1)  # noqa: E731
    rand = lambda: torch.rand(k, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    u = pick(rand() * float(cdf[-1]))
    r = rand()
    c = comm_d[u]
    x = torch.where(rand() < 1.0 - mixing, base_d[c] + r * mass_d[c], r * float(cdf[-1]))
    v = pick(x)
    labels = np.empty(n, np.int32)
    labels[order] = comm
    return _csr(snap, order_d[u][draw], order_d[v][draw], n, T, w_max, seed % 1000003), to(labels)


def _contact(n, T, pool, per_snapshot, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    groups = 9
    size = max(1, n // groups)
    a = torch.randint(0, n, (pool,), generator=gen, device=dev)
    mate = (torch.div(a, size, rounding_mode="floor") * size + torch.randint(0, size, (pool,), generator=gen, device=dev)) % n
    other = torch.randint(0, n, (pool,), generator=gen, device=dev)
    b = torch.where(torch.rand(pool, generator=gen, device=dev) < 0.7, mate, other)
    m = int(T * per_snapshot)
    snap = torch.randint(0, T, (m,), generator=gen, device=dev)
    j = torch.randint(0, pool, (m,), generator=gen, device=dev)
    return _csr(snap, a[j], b[j], n, T, 1, seed % 1000003)


def _graph(case, seed):
    if case["graph"] == "planted":
        return _planted(case["n"], case["T"], case["mean_deg"], case["w_max"], seed)
    if case["graph"] == "powerlaw":
        return _powerlaw(case["n"], case["T"], case["mean_deg"], case["deg_exp"], case["mixing"], case["w_max"], seed)
    return _contact(case["n"], case["T"], case["pool"], case["per_snapshot"], seed), None


# --------------------------------------------------------------------------
# the cases


def _case(call, graph, n, T, name=None, **more):
    c = {"call": call, "graph": graph, "n": n, "T": T}
    if graph == "planted":
        c.update(mean_deg=16.0, w_max=8)
    elif graph == "powerlaw":
        c.update(mean_deg=20.0, deg_exp=2.5, mixing=0.3, w_max=8)
    else:
        c.update(pool=7004, per_snapshot=25.56)
    if call in ("solve", "sweep"):
        c.update(omega_num=1, omega_den=1, gamma_num=1, gamma_den=1, null="multislice", coupling="ordinal",
                 theta_den=0, fresh="", warm=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a kept handle re-solved: every level is a few thousand nodes or less
        _case("solve", "planted", 1000, 4, "solve_small", mean_deg=16.0, w_max=1),
        # the first call of a program: host arrays in, labels out, handle released
        _case("solve", "planted", 2003, 6, "solve_small_new", fresh="host"),
        # the plain benchmark shape
        _case("solve", "powerlaw", 100_000, 16, "solve_t16"),
        # the long benchmark shape, from device arrays, once
        _case("solve", "powerlaw", 100_000, 64, "solve_t64", mean_deg=16.0, deg_exp=2.3, mixing=0.4, w_max=16,
              fresh="device"),
        # randomised refinement
        _case("solve", "powerlaw", 30_011, 12, "solve_random", theta_den=100),
        # Constant Potts Model, every pair of snapshots coupled
        _case("solve", "powerlaw", 12_345, 8, "solve_cpm_cat", null="cpm", coupling="categorical", gamma_num=1,
              gamma_den=100),
        # global null model, warm start
        _case("solve", "planted", 60_000, 8, "solve_global", null="global", warm=True, omega_num=1, omega_den=10),
        # the long contact sequence, from host arrays
        _case("solve", "contact", 327, 7375, "contact_long", fresh="host", w_max=1),
        # windows of 64 snapshots at a stride of 32
        _case("windows", "contact", 327, 320, "windows", W=64, stride=32),
        # 4 graphs x 9 (gamma, omega) in one batch
        _case("sweep", "planted", 8000, 12, "sweep_batch", graphs=4, points=9),
        # 3 live graphs, 10 snapshots each, windows of 8
        _case("serve", "planted", 12_000, 10, "serve", graphs=3, window=8),
        # Q of a labelling, graph in pinned host memory
        _case("score", "powerlaw", 100_000, 16, "score"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "solve", "contact", "windows", "sweep", "serve", "score"])
    if call == "contact":
        return _case("solve", "contact", rng.randint(100, 327), _log(rng, 100, 7000), fresh="host", w_max=1)
    if call == "windows":
        W = rng.randint(8, 64)
        return _case("windows", "contact", rng.randint(100, 327), rng.randint(80, 320), W=W, stride=rng.randint(W // 2, W - 1))
    if call == "sweep":
        return _case("sweep", "planted", _log(rng, 500, 8000), rng.randint(2, 12), graphs=rng.randint(1, 4),
                     points=rng.randint(2, 9), mean_deg=float(rng.randint(8, 32)))
    if call == "serve":
        return _case("serve", "planted", _log(rng, 500, 12_000), rng.randint(6, 10), graphs=rng.randint(1, 3),
                     window=rng.randint(3, 8))
    graph = rng.choice(["planted", "powerlaw"])
    T = rng.randint(2, 32)
    n = _log(rng, 300, min(100_000, (1_600_000 if graph == "powerlaw" else 600_000) // T))
    if call == "score":
        return _case("score", graph, n, T, mean_deg=float(rng.randint(8, 24)))
    num, den = rng.choice([(1, 10), (1, 1), (10, 1), (3, 7)])
    gn, gd = rng.choice([(1, 1), (3, 4), (5, 4), (3, 2)])
    null = rng.choice(["multislice", "multislice", "multislice", "global", "cpm"])
    return _case("solve", graph, n, T, omega_num=num, omega_den=den, gamma_num=gn,
                 gamma_den=gd * 100 if null == "cpm" else gd, null=null, mean_deg=float(rng.randint(8, 24)),
                 coupling="categorical" if T <= 12 and rng.random() < 0.25 else "ordinal",
                 theta_den=100 if rng.random() < 0.2 else 0, fresh=rng.choice(["", "", "device", "host"]),
                 warm=rng.random() < 0.25)


SWEEP_GAMMAS = [(1, 2), (1, 1), (3, 2)]
SWEEP_OMEGAS = [(1, 10), (1, 1), (10, 1)]


def _sub_sizes(case):
    """n and T of the graphs of a sweep or a serving session: from the case's
    n down by halves (odd sizes among them)."""
    return [(max(8, case["n"] // 2 ** i + i), max(2, case["T"] - i) if case["call"] == "sweep" else case["T"])
            for i in range(case["graphs"])]


def prepare(case, seed):
    st = {"case": case}
    call = case["call"]
    if call == "sweep":
        graphs = [_planted(n, T, case["mean_deg"], case["w_max"], seed * 16 + i)[0]
                  for i, (n, T) in enumerate(_sub_sizes(case))]
        st["snaps"] = graphs
        st["handles"] = [mslice.mslice_build(g, device_ptrs=True) for g in graphs]
        return st
    if call == "serve":
        st["streams"] = [[x.host() for x in _planted(n, T, case["mean_deg"], case["w_max"], seed * 16 + i)[0]]
                         for i, (n, T) in enumerate(_sub_sizes(case))]
        return st
    snaps, labels = _graph(case, seed)
    n, T = case["n"], case["T"]
    if call == "windows":
        st["snaps"] = [x.host() for x in snaps]
    elif call == "score":
        st["snaps"] = [x.host(pin=True) for x in snaps]
        st["labels"] = labels.repeat(T).contiguous()
    else:
        if case["fresh"] == "host":
            st["snaps"] = [x.host() for x in snaps]
        else:
            st["snaps"] = snaps
            st["out"] = torch.empty(n * T, dtype=torch.int32, device="cuda")
        st["init"] = None
        if case["warm"]:
            # the labels of an earlier window: the communities, one node in eight moved off
            gen = torch.Generator(device="cuda")
            gen.manual_seed(seed + 7)
            init = labels.repeat(T)
            odd = torch.rand(n * T, generator=gen, device="cuda") < 0.125
            init = torch.where(odd, torch.arange(n * T, device="cuda", dtype=torch.int32), init).contiguous()
            st["init"] = init.cpu().numpy() if case["fresh"] == "host" else init
        if not case["fresh"]:
            st["handle"] = mslice.mslice_build(snaps, omega=(case["omega_num"], case["omega_den"]), device_ptrs=True,
                                               coupling=case["coupling"])
    torch.cuda.synchronize()
    return st


def _solve(h, st):
    case = st["case"]
    labels, Q, _ = h.mslice_leiden(gamma=(case["gamma_num"], case["gamma_den"]),
                                   omega=(case["omega_num"], case["omega_den"]), null=case["null"],
                                   theta=(1, case["theta_den"]) if case["theta_den"] else None, init=st["init"],
                                   out=st.get("out"))
    return {"labels": labels, "Q": Q}


def run(st):
    case = st["case"]
    call = case["call"]
    if call == "solve":
        if not case["fresh"]:
            return _solve(st["handle"], st)
        with mslice.mslice_build(st["snaps"], omega=(case["omega_num"], case["omega_den"]),
                                 device_ptrs=case["fresh"] == "device", coupling=case["coupling"]) as h:
            return _solve(h, st)
    if call == "windows":
        labels, Q, _ = mslice.mslice_leiden_windowed(st["snaps"], case["W"], case["stride"])
        return {"labels": labels, "Q": np.array(Q)}
    if call == "sweep":
        with mslice.Batch() as b:
            for h in st["handles"]:
                for p in range(case["points"]):
                    b.mslice_batch_add(h, gamma=SWEEP_GAMMAS[p // 3], omega=SWEEP_OMEGAS[p % 3])
            b.mslice_batch_run()
            labels, Q = b.mslice_batch_results()
        return {"labels": labels, "Q": Q}
    if call == "serve":
        labels, Q = [], []
        with mslice.Server(window=case["window"]) as srv:
            ids = [srv.mslice_server_add_graph(len(g[0].indptr) - 1) for g in st["streams"]]
            reqs = [srv.mslice_server_submit(i, g[t]) for t in range(case["T"]) for i, g in zip(ids, st["streams"])]
            for r in reqs:
                lab, info = srv.mslice_server_wait(r)
                labels.append(lab)
                Q.append(info["Q"])
        return {"labels": np.concatenate(labels), "Q": np.array(Q)}
    with mslice.mslice_build(st["snaps"], host_tensors=True) as h:
        return {"Q": h.mslice_modularity(st["labels"])}


def _entries(graph, n, T, mean_deg):
    return int(n * T * mean_deg)


def work(case):
    """Bytes of the snapshots (8 a row, 8 an entry) and the labels, each once."""
    call, n, T = case["call"], case["n"], case["T"]
    if call == "sweep":
        b = sum(8 * x * t + 8 * _entries("planted", x, t, case["mean_deg"]) + 4 * x * t * case["points"]
                for x, t in _sub_sizes(case))
    elif call == "serve":
        b = sum(8 * x * t + 8 * _entries("planted", x, t, case["mean_deg"]) + 4 * x * sum(min(k + 1, case["window"]) for k in range(t))
                for x, t in _sub_sizes(case))
    else:
        deg = 2 * case["per_snapshot"] / n if case["graph"] == "contact" else case["mean_deg"]
        b = 8 * n * T + 8 * _entries(case["graph"], n, T, deg) + 4 * n * T
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Q of the labelling in 64 bits, straight from its definition."""
    if case["call"] != "score":
        return None
    snaps, labels = _graph(case, seed)
    n, T = case["n"], case["T"]
    lab = labels.long()
    two_m_all, inside, null = 0.0, 0.0, 0.0
    for s in snaps:
        deg = s.indptr[1:] - s.indptr[:-1]
        row = torch.repeat_interleave(torch.arange(n, device=lab.device), deg)
        w = s.weights.double()
        two_m = float(w.sum())
        if two_m == 0:
            continue
        inside += float(w[lab[row] == lab[s.indices.long()]].sum())
        k = torch.zeros(n, dtype=torch.float64, device=lab.device).index_add_(0, row, w)
        mass = torch.zeros(n, dtype=torch.float64, device=lab.device).index_add_(0, lab, k)
        null += float((mass * mass).sum()) / two_m
        two_m_all += two_m
    coupled = 2.0 * n * (T - 1)  # omega = 1, every copy keeps its label
    two_mu = two_m_all + coupled
    return {"Q": (inside + coupled - null) / two_mu if two_mu else 0.0}
