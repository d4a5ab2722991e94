"""Performance cases of the hypergraph partitioner: what its users have it do.

Inputs follow the repository's workload recipes (Zipf nets with preferential
or uniform pins, uniform nets with geometric sizes, large-net stress, graphs),
drawn on the GPU from the case's seed.  Every case goes through the entry
points of ``paper_2303_17679_gb300.hg``; all results are whole numbers.

Kinds of cases ("kind"):
  partition  hg_create + hg_partition + hg_destroy: one hypergraph in, its
             partition and objective out (host or device arrays)
  batch      many small hypergraphs through the executor, host arrays in,
             partitions out
  coarsen    one clustering and contraction step on a handle that is kept,
             its node map and sizes
  refine     label propagation of a given partition on a handle that is kept
  gains      the refinement tools on a handle that is kept: gain table, a
             set of moves applied to it, exact gains of the move sequence
  objective  the allocation-free objective of a partition of device arrays
"""
import math
import os
import types

import numpy as np

# Streams of the executor's slots share hardware queues unless the process
# asks for more of them before CUDA starts (include/hg.h).
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import torch  # noqa: E402

from paper_2303_17679_gb300 import hg  # noqa: E402

EPS_PPM, PASSES = 30000, 5
SLOTS = 16


def listed():
    return [
        # the smallest call: scoring a partition inside a serving loop (n = m = 10,000 uniform)
        dict(name="objective_10k", kind="objective", gen="uniform", n=10_000, m=10_000, k=2),
        # plain single level: label propagation of the n = m = 10,000 uniform hypergraph
        dict(name="refine_10k_k2", kind="refine", gen="uniform", n=10_000, m=10_000, k=2),
        # the smallest serving request, 10,000 pins from host arrays
        dict(name="partition_serve_10k_k8", kind="partition", gen="serve", n=1_471, m=1_471, k=8,
             host=True, communities=False),
        # a middling serving request, 141,000 pins from host arrays
        dict(name="partition_serve_141k_k32", kind="partition", gen="serve", n=20_797, m=20_797,
             k=32, host=True, communities=False),
        # one batch of small and middling instances through the executor
        dict(name="batch_32", kind="batch", count=32, n_lo=1_000, n_hi=50_000),
        # the benchmark's whole V-cycle: n = m = 1e6 Zipf nets, heavy-tailed degrees
        dict(name="partition_zipf_1m_k8", kind="partition", gen="zipf", n=1_000_000, m=1_000_000,
             k=8, host=False, communities=False),
        # the largest: 4e6 nodes, 1 % nets of a thousand pins and more, k = 64
        dict(name="partition_largenet_4m_k64", kind="partition", gen="largenet", n=4_000_000,
             m=2_000_000, k=64, host=False, communities=False),
        # a graph (nets of two pins) on the graph path
        dict(name="partition_graph_1m_k8", kind="partition", gen="graph", n=1_000_000, m=4_000_000,
             k=8, host=False, communities=False),
        # communities detected first, odd sizes, nodes outnumber nets
        dict(name="partition_communities_250k_k4", kind="partition", gen="zipf", n=250_007,
             m=199_999, k=4, host=False, communities=True),
        # one clustering and contraction step alone
        dict(name="coarsen_zipf_500k_k16", kind="coarsen", gen="zipf", n=500_009, m=750_011, k=16),
        # refinement of a given partition on a large level
        dict(name="refine_zipf_500k_k16", kind="refine", gen="zipf", n=500_009, m=499_979, k=16),
        # gain table, moves and exact gains of a tenth of the nodes
        dict(name="gains_zipf_1m_k8", kind="gains", gen="zipf", n=1_000_000, m=1_000_000, k=8,
             moves=100_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["partition"] * 5 + ["batch", "coarsen", "refine", "refine", "gains",
                                          "objective"])
    if kind == "batch":
        lo = _log_int(rng, 1_000, 5_000)
        return dict(kind=kind, count=rng.randint(8, 48), n_lo=lo, n_hi=_log_int(rng, 2 * lo, 60_000))
    gen = rng.choice(["zipf", "zipf", "serve", "uniform", "graph", "largenet"])
    k = rng.choice([2, 4, 8, 16, 32, 64]) if rng.random() < 0.8 else rng.randint(2, 64)
    if gen == "largenet":
        n = _log_int(rng, 200_000, 3_500_000)
        m = int(n * rng.uniform(0.3, 0.5))
    elif gen == "graph":
        n = _log_int(rng, 3_000, 900_000)
        m = int(n * rng.uniform(2.0, 4.5))
    else:
        n = _log_int(rng, 1_471, 900_000)
        m = n if gen == "serve" else max(1_000, int(n * rng.uniform(0.5, 2.0)))
        m = min(m, 1_000_000)
    c = dict(kind=kind, gen=gen, n=n, m=m, k=k)
    if kind == "partition":
        c["host"] = rng.random() < 0.5
        c["communities"] = gen != "largenet" and rng.random() < 0.2
    if kind == "coarsen":  # at most 160 k nodes are not coarsened any further
        c["k"] = max(2, min(k, n // 640))
    if kind == "gains":
        c["moves"] = max(1, int(n * rng.uniform(0.01, 0.3)))
    return c


# ----------------------------------------------------------------- inputs

ZIPF_S, ZIPF_LO, ZIPF_HI = 2.2, 2, 1024


def _zipf_law():
    x = np.arange(ZIPF_LO, ZIPF_HI + 1, dtype=np.float64)
    w = x ** -ZIPF_S
    return np.cumsum(w) / w.sum(), float((x * w).sum() / w.sum())


def _rand(g, count):
    return torch.rand(count, generator=g, device="cuda", dtype=torch.float64)


def _below(u, bound):
    """Whole numbers in [0, bound) from uniforms in [0, 1)."""
    return torch.minimum((u * bound).long(), torch.as_tensor(bound, device=u.device) - 1)


def _sizes(gen, n, m, g):
    if gen == "graph":
        return torch.full((m,), 2, dtype=torch.int64, device="cuda")
    u = _rand(g, m)
    if gen in ("zipf", "serve"):
        cdf = torch.from_numpy(_zipf_law()[0]).cuda()
        s = ZIPF_LO + torch.searchsorted(cdf, u, right=True)
        return s.clamp(max=min(ZIPF_HI, n))
    s = 2 + torch.floor(torch.log(1.0 - u) / math.log(0.7)).long()  # 2 + Geom(0.3)
    if gen == "uniform":
        return s.clamp(max=min(64, n))
    s = s.clamp(max=16)  # large nets: every 100th of size density x^-4 on [1000, 100000]
    big = torch.arange(0, m, 100, device="cuda")
    hi = float(min(100_000, n))
    a, b = 1000.0 ** -3, hi ** -3
    s[big] = torch.floor((a + u[big] * (b - a)) ** (-1.0 / 3.0)).long().clamp(1000, int(hi))
    s[0] = int(hi)
    return s


def _pins(gen, n, p, g):
    if gen in ("serve", "uniform", "largenet"):
        return _below(_rand(g, p), n)
    # preferential: pin i is a fresh node (the next of a permutation) with
    # probability n / (n + i), else a copy of a uniformly chosen earlier pin;
    # the chains of copies are followed by pointer doubling
    i = torch.arange(p, device="cuda")
    fresh = _rand(g, p) * (n + i) < n
    fresh[0] = True
    parent = torch.where(fresh, i, _below(_rand(g, p), i.clamp(min=1)))
    while True:
        up = parent[parent]
        if torch.equal(up, parent):
            break
        parent = up
    rank = torch.cumsum(fresh.long(), 0) - 1
    perm = torch.randperm(n, generator=g, device="cuda")
    node = torch.where(rank < n, perm[rank.clamp(max=n - 1)], _below(_rand(g, p), n))
    return node[parent]


def _hypergraph(gen, n, m, seed):
    """Device CSR (int32): offsets, pins, net weights, node weights; a node
    drawn twice in a net is kept once (a graph's loop gets another end)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    sizes = _sizes(gen, n, m, g)
    p = int(sizes.sum())
    net = torch.repeat_interleave(torch.arange(m, device="cuda"), sizes)
    pins = _pins(gen, n, p, g)
    if gen == "graph":
        e = pins.view(m, 2)
        e[:, 1] = torch.where(e[:, 0] == e[:, 1], (e[:, 1] + 1) % n, e[:, 1])
    else:
        key, order = torch.sort(net * n + pins, stable=True)
        twice = torch.zeros(p, dtype=torch.bool, device="cuda")
        twice[order[1:]] = key[1:] == key[:-1]
        net, pins = net[~twice], pins[~twice]
    off = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(net, minlength=m), 0)
    top_w = {"zipf": 10, "graph": 10, "uniform": 10, "largenet": 100, "serve": 1}[gen]
    top_c = {"zipf": 10, "graph": 10, "uniform": 10, "largenet": 1, "serve": 1}[gen]
    w = 1 + _below(_rand(g, m), top_w)
    c = 1 + _below(_rand(g, n), top_c)
    return types.SimpleNamespace(n=n, m=m, p=int(pins.numel()), offsets=off.int(),
                                 pins=pins.int(), net_w=w.int(), node_w=c.int())


def _to_host(x):
    return types.SimpleNamespace(n=x.n, m=x.m, p=x.p, offsets=x.offsets.cpu().numpy(),
                                 pins=x.pins.cpu().numpy(), net_w=x.net_w.cpu().numpy(),
                                 node_w=x.node_w.cpu().numpy())


def _batch(case, seed):
    """Instances with n log-uniform in [n_lo, n_hi], m / n in [0.5, 3], uniform
    nets, k in {2, 4, 8, 16, 32}; the case fixes their sizes, the seed the rest."""
    r = np.random.default_rng([case["count"], case["n_lo"], case["n_hi"]])
    jobs = []
    for i in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        m = max(1, int(round(n * r.uniform(0.5, 3.0))))
        k = int(r.choice([2, 4, 8, 16, 32]))
        jobs.append((_to_host(_hypergraph("uniform", n, m, seed * 1_000 + i)), k))
    return jobs


# ------------------------------------------------------------------ states

class _Handle:
    """A library handle that is destroyed with its state."""

    def __init__(self, x, opt):
        self.h = hg.hg_create(x.n, x.m, x.offsets, x.pins, x.net_w, x.node_w, hg.HG_MEM_DEVICE,
                              opt, torch.cuda.current_stream())

    def __del__(self):
        hg.hg_destroy(self.h)


class _Slots:
    """An executor that is closed with its state."""

    def __init__(self):
        self.ex = hg.Executor(SLOTS)

    def __del__(self):
        self.ex.close()


def _options(case, seed):
    o = hg.hg_default_options()
    o.seed = seed & 0xFFFFFFFF
    o.community_detection = 1 if case.get("communities") else 0
    return o


def prepare(case, seed):
    if case["kind"] == "batch":
        return dict(case=case, jobs=_batch(case, seed), slots=_Slots())
    x = _hypergraph(case["gen"], case["n"], case["m"], seed)
    s = dict(case=case, x=x, opt=_options(case, seed))
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    k, n = case["k"], case["n"]
    if case["kind"] == "partition":
        if case["host"]:
            s["x"] = _to_host(x)
        s["part"] = torch.empty(n, dtype=torch.int32, device="cuda")
        return s
    if case["kind"] != "objective":
        s["handle"] = _Handle(x, s["opt"])
    if case["kind"] == "coarsen":
        return s
    s["part0"] = _below(_rand(g, n), k).int()
    if case["kind"] == "gains":
        nodes = torch.randperm(n, generator=g, device="cuda")[:case["moves"]]
        step = 1 + _below(_rand(g, nodes.numel()), k - 1)
        s["nodes"] = nodes.int()
        s["targets"] = ((s["part0"][nodes] + step) % k).int()
        s["benefit"] = torch.empty(n, dtype=torch.int64, device="cuda")
        s["penalty"] = torch.empty((n, k), dtype=torch.int64, device="cuda")
        s["gains"] = torch.empty(nodes.numel(), dtype=torch.int64, device="cuda")
    return s


# ------------------------------------------------------------------ passes

def _run_partition(s):
    c, x = s["case"], s["x"]
    h = hg.hg_create(x.n, x.m, x.offsets, x.pins, x.net_w, x.node_w,
                     hg.HG_MEM_HOST if c["host"] else hg.HG_MEM_DEVICE, s["opt"],
                     torch.cuda.current_stream())
    try:
        obj = hg.hg_partition(h, c["k"], EPS_PPM, PASSES, s["part"])
        levels = hg.hg_num_levels(h)
    finally:
        hg.hg_destroy(h)
    return dict(part=s["part"], objective=obj, levels=levels)


def _run_batch(s):
    ex, jobs = s["slots"].ex, s["jobs"]
    for i in sorted(range(len(jobs)), key=lambda i: -jobs[i][0].p):
        ex.submit(jobs[i][0], jobs[i][1], EPS_PPM, PASSES, tag=i)
    got = {}
    while len(got) < len(jobs):
        for r in ex.wait():
            got[r["tag"]] = r
    return dict(parts=np.concatenate([got[i]["part"] for i in range(len(jobs))]),
                objectives=np.array([got[i]["objective"] for i in range(len(jobs))]),
                status=np.array([got[i]["status"] for i in range(len(jobs))]))


def _run_coarsen(s):
    h, k, n = s["handle"].h, s["case"]["k"], s["case"]["n"]
    hg.hg_truncate(h, 0)
    status, level, n2, m2, p2 = hg.hg_coarsen_level(h, k)
    if status != hg.HG_OK:
        return dict(status=status)
    # the coarse node of every node, and the cut of a partition of the coarse nodes
    ids = torch.arange(n2, dtype=torch.int32, device="cuda")
    node_map = torch.empty(n, dtype=torch.int32, device="cuda")
    hg.hg_project(h, level, ids, node_map)
    return dict(status=status, n=n2, m=m2, p=p2, map=node_map,
                objective=hg.hg_objective(h, level, k, ids % k))


def _run_refine(s):
    part = s["part0"].clone()
    obj, moves = hg.hg_lp_refine(s["handle"].h, 0, s["case"]["k"], EPS_PPM, PASSES, part)
    return dict(part=part, objective=obj, moves=moves)


def _run_gains(s):
    h, k = s["handle"].h, s["case"]["k"]
    hg.hg_recalculate_gains(h, 0, k, s["part0"], s["nodes"], s["targets"], s["gains"])
    part = s["part0"].clone()
    hg.hg_gain_table(h, 0, k, part, s["benefit"], s["penalty"])
    hg.hg_gain_table_move(h, 0, k, part, s["nodes"], s["targets"], s["benefit"], s["penalty"])
    return dict(gains=s["gains"], part=part, benefit=s["benefit"], penalty=s["penalty"])


def _run_objective(s):
    x = s["x"]
    obj, bw = hg.hg_objective_noalloc(x.n, x.m, x.p, x.offsets, x.pins, x.net_w, x.node_w,
                                      s["case"]["k"], s["part0"], torch.cuda.current_stream())
    return dict(objective=obj, block_weights=bw)


_RUN = dict(partition=_run_partition, batch=_run_batch, coarsen=_run_coarsen, refine=_run_refine,
            gains=_run_gains, objective=_run_objective)


def run(state):
    return _RUN[state["case"]["kind"]](state)


# -------------------------------------------------------------------- work

def _mean_size(gen):
    if gen in ("zipf", "serve"):
        return _zipf_law()[1]
    return {"graph": 2.0, "uniform": 2 + 0.7 / 0.3, "largenet": 0.99 * 4.3 + 0.01 * 1500}[gen]


def _csr_bytes(gen, n, m):
    return 4.0 * (m * _mean_size(gen) + 2 * m + n)


def work(case):
    """The input arrays read once, the outputs written once (all 4 bytes, the
    gain table and gains 8), and one integer add per pin."""
    if case["kind"] == "batch":
        n = case["count"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        m = 1.75 * n
        return dict(bytes=_csr_bytes("uniform", n, m) + 4 * n, flops=m * _mean_size("uniform"))
    n, m, k = case["n"], case["m"], case["k"]
    b = _csr_bytes(case["gen"], n, m)
    if case["kind"] in ("partition", "coarsen"):
        b += 4 * n
    elif case["kind"] == "refine":
        b += 8 * n
    elif case["kind"] == "gains":
        b += 8 * n + 8.0 * n * (k + 1) + 16 * case["moves"]
    else:
        b += 4 * n
    return dict(bytes=b, flops=m * _mean_size(case["gen"]))


# ------------------------------------------------------------------- exact

def _pin_counts(x, part, k):
    net = torch.repeat_interleave(torch.arange(x.m, device="cuda"), (x.offsets[1:] - x.offsets[:-1]).long())
    phi = torch.zeros(x.m * k, dtype=torch.int64, device="cuda")
    phi.index_add_(0, net * k + part[x.pins.long()].long(), torch.ones_like(net))
    return net, phi.view(x.m, k)


def _exact_gains(s):
    """Gains of the sequence from the first move into, the last move out of
    and the unmoved pins of every block of every net; the gain table of the
    partition after the moves from its pin counts."""
    x, k, m, n = s["x"], s["case"]["k"], s["case"]["m"], s["case"]["n"]
    nodes, targets, l = s["nodes"].long(), s["targets"].long(), s["nodes"].numel()
    part, pins, w = s["part0"].long(), x.pins.long(), x.net_w.long()
    net, _ = _pin_counts(x, part, k)
    idx = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    idx[nodes] = torch.arange(l, device="cuda")
    i = idx[pins]
    moved = i >= 0
    out_slot = net * k + part[pins]
    in_slot = (net * k)[moved] + targets[i[moved]]
    first_in = torch.full((m * k,), l, dtype=torch.int64, device="cuda")
    first_in.scatter_reduce_(0, in_slot, i[moved], "amin")
    last_out = torch.full((m * k,), -1, dtype=torch.int64, device="cuda")
    last_out.scatter_reduce_(0, out_slot[moved], i[moved], "amax")
    stay = torch.zeros(m * k, dtype=torch.int64, device="cuda")
    stay.index_add_(0, out_slot[~moved], torch.ones_like(out_slot[~moved]))
    im, o = i[moved], out_slot[moved]
    wm = w[net[moved]]
    won = (last_out[o] == im) & (im < first_in[o]) & (stay[o] == 0)
    lost = (first_in[in_slot] == im) & (im > last_out[in_slot]) & (stay[in_slot] == 0)
    gains = torch.zeros(l, dtype=torch.int64, device="cuda")
    gains.index_add_(0, im, wm * won.long() - wm * lost.long())
    after = part.clone()
    after[nodes] = targets
    net, phi = _pin_counts(x, after, k)
    benefit = torch.zeros(n, dtype=torch.int64, device="cuda")
    benefit.index_add_(0, pins, w[net] * (phi[net, after[pins]] == 1).long())
    penalty = torch.stack([torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(
        0, pins, w[net] * (phi[net, b] == 0).long()) for b in range(k)], dim=1)
    return dict(gains=gains, part=after.int(), benefit=benefit, penalty=penalty.contiguous())


def exact(case, seed):
    """The same results from plain torch for the objective and the gains; the
    multilevel results, the refinement and the clustering are whole numbers
    decided move by move, which plain torch takes minutes for."""
    if case["kind"] not in ("objective", "gains"):
        return None
    s = prepare(case, seed)
    if case["kind"] == "gains":
        return _exact_gains(s)
    x, k = s["x"], case["k"]
    _, phi = _pin_counts(x, s["part0"], k)
    lam = (phi > 0).sum(1)
    bw = torch.zeros(k, dtype=torch.int64, device="cuda").index_add_(0, s["part0"].long(),
                                                                    x.node_w.long())
    return dict(objective=int(((lam - 1).clamp(min=0) * x.net_w.long()).sum()), block_weights=bw.cpu().numpy())
