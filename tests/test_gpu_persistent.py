"""The persistent kernels on the GPU: barriers behind loops that the lanes of a
warp leave at different times, and what the launch rules decide.  All results are
integers and compared exactly with the oracle."""
import threading

import numpy as np
import pytest

import synth
from tests import hostcc
from tests.tiny import from_nets

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2303_17679_gb300 import build, hg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def create(hgr, seed, S=16, factor=160, **options):
    o = hg.hg_default_options()
    o.seed, o.subrounds, o.contraction_limit_factor = seed, S, factor
    for name, value in options.items():
        setattr(o, name, value)
    return hg.hg_create(hgr.n, hgr.m, hgr.offsets, hgr.pins, hgr.net_w, hgr.node_w,
                        hg.HG_MEM_HOST, o, torch.cuda.current_stream())


# 2 S list counters that are no multiple of a warp, node counts that are none of a
# block: small levels, whose blocks meet at the barrier of one cluster
@pytest.mark.parametrize("n,S,k", [(333, 1, 2), (1471, 3, 5), (2999, 7, 33), (4001, 33, 8)])
def test_ragged_small_levels(oracle_mod, n, S, k):
    hgr = synth.zipf_preferential(n, n, n, name="ragged")
    vc = oracle_mod.multilevel(hgr, k, 30000, S=S, factor=10, seed=n, max_passes=3)
    h = create(hgr, n, S, 10)
    try:
        part = torch.empty(n, dtype=torch.int32, device="cuda")
        obj = hg.hg_partition(h, k, 30000, 3, part)
        assert hg.hg_num_levels(h) == len(vc.levels)
        assert np.array_equal(part.cpu().numpy(), vc.parts[0]) and obj == vc.objectives[0]
    finally:
        hg.hg_destroy(h)


class Hooks:
    """A caller's allocator whose blocks start `shift` bytes into torch's."""

    def __init__(self, shift):
        self.shift, self.live = shift, {}
        self.alloc, self.free = hg.ALLOC_FN(self.get), hg.FREE_FN(self.put)

    def get(self, size, ctx):
        t = torch.empty(size + self.shift, dtype=torch.uint8, device="cuda")
        self.live[t.data_ptr() + self.shift] = t
        return t.data_ptr() + self.shift

    def put(self, ptr, ctx):
        del self.live[ptr]

    def options(self):
        return dict(dev_alloc=self.alloc, dev_free=self.free)


# k = 64: net records of 32 bytes; nets of two pins: pins read in pairs
@pytest.mark.parametrize("shift", [0, 4, 8, 16])
@pytest.mark.parametrize("graph,k", [(False, 64), (False, 8), (True, 64)])
def test_hook_blocks_of_any_alignment(oracle_mod, shift, graph, k):
    hgr = synth.graph_preferential(3, 4000, 20_000) if graph else synth.zipf_preferential(3, 4000, 4000)
    vc = oracle_mod.multilevel(hgr, k, 30000, S=16, factor=10, seed=3, max_passes=3)
    hooks = Hooks(shift)
    h = create(hgr, 3, factor=10, **hooks.options())
    try:
        part = torch.empty(hgr.n, dtype=torch.int32, device="cuda")
        obj = hg.hg_partition(h, k, 30000, 3, part)
        assert np.array_equal(part.cpu().numpy(), vc.parts[0]) and obj == vc.objectives[0]
        b = torch.zeros(hgr.n, dtype=torch.int64, device="cuda")
        p = torch.zeros((hgr.n, k), dtype=torch.int64, device="cuda")
        hg.hg_gain_table(h, 0, k, part, b, p)
        wb, wp = oracle_mod.gain_table(hgr, k, vc.parts[0])
        assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
    finally:
        hg.hg_destroy(h)
    assert not hooks.live


@pytest.mark.parametrize("S", [1, 16])
def test_louvain_hubs(oracle_mod, S):
    """Net vertices around the degrees where a vertex is split into parts and into
    chunks of its edges, and a node vertex above both."""
    n = 60_000
    rng = np.random.default_rng(S)
    sizes = [4096, 4097, 32_767, 32_768, 32_769, 33_792, 33_793, 50_000]
    nets = [rng.choice(n, size=s, replace=False).tolist() for s in sizes]
    nets += [[7, int(v)] for v in rng.choice(np.arange(8, n), size=40_000, replace=False)]
    nets += rng.integers(0, n // 2, size=(20_000, 1)).repeat(2, 1).__add__([0, n // 2]).tolist()
    hgr = from_nets(n, nets, rng.integers(1, 9, size=len(nets)), None)
    want, levels, moves = oracle_mod.communities(hgr, S=S, seed=2)
    h = create(hgr, 2, S)
    try:
        hg.hg_detect_communities(h)
        assert np.array_equal(hg.hg_get_communities(h, 0), want)
        st = hg.hg_get_stats(h)
        assert st["louvain_levels"] == levels and st["louvain_moves"] == moves
    finally:
        hg.hg_destroy(h)


# A barrier of two blocks with a short limit.  late: block 1 arrives after about
# 50 ms, reporting its progress or not; never: it leaves without arriving.
@pytest.mark.parametrize("late,beats,passes", [(0, 0, 1), (1, 1, 1), (1, 0, 0), (2, 0, 0)])
def test_barrier_gives_up_on_lack_of_progress(tmp_path, late, beats, passes):
    hostcc.run(tmp_path, ["gridsync.cuh"], f"""
    using namespace hgk;
    __global__ void k_wait(unsigned* barrier, int32_t* status, int32_t* passed) {{
      unsigned gen = 0;
      if (blockIdx.x == 1) {{
        if ({late} == 2) return;
        const unsigned long long t0 = now_ns();
        for (int i = 0; {late} == 1 && i < 1 << 20 && now_ns() - t0 < 50000000ull; ++i) {{
          __nanosleep(1000);
          if ({beats} && threadIdx.x == 0) beat(barrier);
        }}
      }}
      if (!grid_sync(false, barrier, status, gen, 1 << 12)) return;
      if (blockIdx.x == 0 && threadIdx.x == 0) *passed = 1;
    }}
    int main() {{
      int32_t* d = nullptr;
      CHECK(cudaMalloc(&d, 16) == cudaSuccess && cudaMemset(d, 0, 16) == cudaSuccess);
      Ctx cx;
      launch_persistent(cx, k_wait, 2, 64, 0, false, (unsigned*)d, d + 2, d + 3);
      int32_t h[4];
      CHECK(cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost) == cudaSuccess);
      CHECK(h[3] == {passes});
      CHECK(h[2] == ({passes} ? DEV_OK : DEV_TIMEOUT));
      return 0;
    }}
    """)


def test_plain_handles_at_once(oracle_mod):
    """Levels of every launch form from several host threads, each result that of
    the call alone."""
    jobs = [(synth.zipf_preferential(i, n, n), k) for i, (n, k) in
            enumerate([(1500, 2), (5000, 40), (12_000, 8), (20_000, 4)])]
    want = [oracle_mod.multilevel(g, k, 30000, S=16, factor=20, seed=5, max_passes=2)
            for g, k in jobs]
    got = [None] * len(jobs)

    def work(i):
        g, k = jobs[i]
        o = hg.hg_default_options()
        o.seed, o.contraction_limit_factor, o.blocking_sync = 5, 20, i % 2
        st = torch.cuda.Stream()
        for _ in range(6):
            part = torch.empty(g.n, dtype=torch.int32, device="cuda")
            st.wait_stream(torch.cuda.default_stream())
            h = hg.hg_create(g.n, g.m, g.offsets, g.pins, g.net_w, g.node_w, hg.HG_MEM_HOST, o, st)
            try:
                obj = hg.hg_partition(h, k, 30000, 2, part)
            finally:
                hg.hg_destroy(h)
            same = np.array_equal(part.cpu().numpy(), want[i].parts[0])
            got[i] = (obj, same) if got[i] in (None, (obj, same)) else "differs"

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert got == [(w.objectives[0], True) for w in want]


def test_handles_after_a_device_reset(tmp_path):
    """The same thread and the same kernels, with the caller's own allocator: what
    the library keeps beyond a handle must not outlive the context."""
    out = hostcc.run(tmp_path, ["hg.h"], """
    void* get(size_t bytes, void*) {
      void* p = nullptr;
      return cudaMalloc(&p, bytes) == cudaSuccess ? p : nullptr;
    }
    void put(void* p, void*) { cudaFree(p); }
    uint64_t partition() {
      const int n = 12000, m = 12000;  // levels with the wide shared-memory forms
      std::vector<int32_t> off{0}, pins;
      uint32_t x = 1;
      for (int e = 0; e < m; ++e) {
        const int size = 2 + e % 5 + (e % 500 == 0 ? 1500 : 0);
        const int at = (x = x * 1664525u + 1013904223u) % n;
        for (int i = 0; i < size; ++i) pins.push_back((at + i * 7) % n);
        off.push_back((int32_t)pins.size());
      }
      hg_options o;
      hg_default_options(&o);
      o.dev_alloc = get;
      o.dev_free = put;
      o.contraction_limit_factor = 20;
      o.community_detection = 1;
      hg_t* h = nullptr;
      CHECK(hg_create(n, m, off.data(), pins.data(), nullptr, nullptr, HG_MEM_HOST, &o, nullptr,
                      &h) == HG_OK);
      int32_t* part = nullptr;
      CHECK(cudaMalloc(&part, 4 * n) == cudaSuccess);
      int64_t f = 0;
      CHECK(hg_partition(h, 4, 30000, 3, part, &f) == HG_OK);
      std::vector<int32_t> got(n);
      CHECK(cudaMemcpy(got.data(), part, 4 * n, cudaMemcpyDeviceToHost) == cudaSuccess);
      hg_destroy(h);
      cudaFree(part);
      uint64_t sum = (uint64_t)f;
      for (int32_t b : got) sum = sum * 31 + (uint64_t)b;
      return sum;
    }
    int main() {
      const uint64_t before = partition();
      for (int i = 0; i < 2; ++i) {
        CHECK(cudaDeviceReset() == cudaSuccess);
        CHECK(partition() == before);
      }
      std::printf("same %llu", (unsigned long long)before);
      return 0;
    }
    """, link=[build.LIB, "-cudart", "shared", "-Xlinker", "-rpath", "-Xlinker", build.HERE])
    assert out.startswith("same")


def mix64(x):
    """SplitMix64's output function on a uint64 array."""
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def part_of(ids, parts):
    """The part of a candidate (rating.cuh)."""
    h = (ids.astype(np.uint64) * np.uint64(0x85EBCA77)) & np.uint64(0xffffffff)
    return (h * np.uint64(parts)) >> np.uint64(32)


# A node rated in the first sub-round, before anything has joined, with candidates
# that all lie in one part of the table: 2-pin nets (64-bit ratings, 16384 slots) on
# the hypergraph and the graph path, nets of 750 pins (32-bit, 22528 slots).
@pytest.mark.parametrize("form,count,parts", [("nets", 24_000, 5), ("graph", 24_000, 3),
                                              ("wide nets", 30_000, 3)])
def test_candidates_that_meet_in_one_part(oracle_mod, form, count, parts):
    n, seed = 200_000, 1
    ids = np.arange(n, dtype=np.uint64)
    hub = int(np.flatnonzero(mix64(ids ^ np.uint64(seed)) % np.uint64(16) == 0)[0])
    cand = np.flatnonzero(part_of(ids, parts) == 0)
    cand = cand[cand != hub][:count]
    assert len(cand) == count and count * 15 // 16 > (22_528 if form == "wide nets" else 16_384)
    if form == "wide nets":
        nets = [[hub, *c.tolist()] for c in cand.reshape(-1, 750)]
    else:
        nets = [[hub, int(v)] for v in cand]
    if form == "nets":
        nets.append([n - 3, n - 2, n - 1])
    rng = np.random.default_rng(2)
    hgr = from_nets(n, nets, rng.integers(1, 100, size=len(nets)), None)
    ref = oracle_mod.multilevel(hgr, 2, 30000, S=16, factor=160, seed=seed, max_passes=0)
    h = create(hgr, seed)
    try:
        assert hg.hg_level_is_graph(h, 0) == (form == "graph")
        assert hg.hg_coarsen_level(h, 2)[0] == hg.HG_OK
        assert np.array_equal(hg.hg_get_level(h, 0, with_map=True)["map"], ref.maps[0])
    finally:
        hg.hg_destroy(h)


def test_louvain_clusters_that_meet_in_one_part(oracle_mod):
    """A net vertex of 32,768 neighbours, sixteen parts, whose clusters all belong to
    one of them."""
    n, size, seed = 700_000, 32_768, 4
    ids = np.arange(n, dtype=np.uint64)
    part = ((mix64(ids ^ np.uint64(0xA5A5A5A500000000)) >> np.uint64(32)) * np.uint64(16)) >> np.uint64(32)
    pins = np.flatnonzero(part == 3)[:size]
    key = seed ^ (1 << 62) ^ (1 << 48) ^ n  # the net's vertex in the first round
    assert len(pins) == size and mix64(np.array([key], np.uint64))[0] % np.uint64(16) < 11
    hgr = from_nets(n, [pins.tolist(), [0, 1], [1, 2, 3]], [100, 1, 1], None)
    want, levels, moves = oracle_mod.communities(hgr, S=16, seed=seed)
    h = create(hgr, seed)
    try:
        hg.hg_detect_communities(h)
        assert np.array_equal(hg.hg_get_communities(h, 0), want)
        st = hg.hg_get_stats(h)
        assert st["louvain_levels"] == levels and st["louvain_moves"] == moves
    finally:
        hg.hg_destroy(h)


def test_phase_times_of_label_propagation():
    hgr = synth.zipf_preferential(1, 200_000, 200_000)
    h = create(hgr, 1)
    try:
        part = torch.empty(hgr.n, dtype=torch.int32, device="cuda")
        hg.hg_initial_partition(h, 0, 4, part)
        hg.hg_enable_timing(h, 1)
        hg.hg_lp_refine(h, 0, 4, 30000, 2, part)
        st = hg.hg_get_stats(h)
        for name in ("ms_phi", "ms_lp_gain", "ms_lp_select", "ms_lp_apply", "ms_objective"):
            assert st[name] > 0, name
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("size,launches", [(20, 0), (4, 1)])
def test_rating_launches_counts_launches(size, launches):
    """Levels without a rated net launch no rating kernel."""
    n = 2000
    hgr = from_nets(n, np.arange(n).reshape(-1, size).tolist())
    h = create(hgr, 1, factor=10, rating_max_net_size=10)
    try:
        hg.hg_coarsen_level(h, 2)
        assert hg.hg_get_stats(h)["rating_launches"] == launches
    finally:
        hg.hg_destroy(h)


# hg_create refuses total net or node weights of 2^31 and more, which is what makes
# 32-bit sums enough; a node in every net, many nets (one item per 128 to 1024 of
# them) and few
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("m,k", [(7, 2), (3000, 8), (3000, 40), (40, 33)])
def test_largest_total_weights(oracle_mod, m, k, graph):
    n, top = 4000, (1 << 31) - 1
    rng = np.random.default_rng(m + k)
    size = 2 if graph else 4
    nets = [[0, *rng.choice(np.arange(1, n), size=size - 1, replace=False).tolist()]
            for _ in range(m)]

    def spread(count):
        w = np.full(count, top // count, np.int64)
        w[-1] += top - w.sum()
        return w.astype(np.int32)

    hgr = from_nets(n, nets, spread(m), spread(n))
    assert hgr.net_w.sum(dtype=np.int64) == top == hgr.node_w.sum(dtype=np.int64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()  # noqa: E731
    for part0 in (rng.integers(0, k, size=n).astype(np.int32),
                  np.where(np.arange(n) == 0, 1, 0).astype(np.int32)):
        ref = oracle_mod.lp_refine(hgr, k, part0, 10**9, 16, 3, 0, 3)
        h = create(hgr, 3, lp_block_min_deg=64)
        try:
            d = dev(part0)
            assert hg.hg_lp_refine(h, 0, k, 10**9, 3, d) == (ref["objective"], ref["moves"])
            assert np.array_equal(d.cpu().numpy(), ref["part"])
            b = torch.zeros(n, dtype=torch.int64, device="cuda")
            p = torch.zeros((n, k), dtype=torch.int64, device="cuda")
            hg.hg_gain_table(h, 0, k, dev(part0), b, p)
            wb, wp = oracle_mod.gain_table(hgr, k, part0)
            assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
            hg.hg_initial_partition(h, 0, k, d)
            assert np.array_equal(d.cpu().numpy(), oracle_mod.initial_partition(hgr.node_w, k, 3))
        finally:
            hg.hg_destroy(h)


@pytest.mark.parametrize("k", [9, 32])
def test_directions_longer_than_the_shared_buffers(oracle_mod, k):
    """For k > 8 the selection sorts up to 2048 moves of a direction in shared memory.
    More come from the direction's key list and the overflow list into global keys at
    twice the direction's offset, with their weight prefixes.  All moves are between
    blocks 0 and 1."""
    n, seed, eps = 400_000, 7, 2_000_000_000
    hgr = synth.random_uniform(61 + k, n, n)
    part0 = synth.uniform_ints(n + k, n, 0, 1)
    _, mv = oracle_mod.lp_subround(hgr, k, part0, eps, 16, seed, 0, 0, 0)
    assert np.bincount(mv["src"] * k + mv["dst"], minlength=k * k).max() > 2048
    ref = oracle_mod.lp_refine(hgr, k, part0, eps, 16, seed, 0, 1)
    h = create(hgr, seed)
    try:
        d = torch.from_numpy(np.ascontiguousarray(part0, np.int32)).cuda()
        assert hg.hg_lp_refine(h, 0, k, eps, 1, d) == (ref["objective"], ref["moves"])
        assert np.array_equal(d.cpu().numpy(), ref["part"])
    finally:
        hg.hg_destroy(h)


def nets_around(n, sizes, seed, rest=3000):
    """A net of each size and `rest` nets of three pins."""
    rng = np.random.default_rng(seed)
    nets = [rng.choice(n, size=s, replace=False).tolist() for s in sizes]
    nets += [rng.choice(n, size=3, replace=False).tolist() for _ in range(rest)]
    order = rng.permutation(len(nets))
    return from_nets(n, [nets[i] for i in order], rng.integers(1, 9, size=len(nets)),
                     rng.integers(1, 4, size=n))


# nets around the size above which a block, or on levels of more than 131,072 pins the
# grid by chunks, counts a net
@pytest.mark.parametrize("sizes,rest", [([2048, 2049, 4096, 4097, 8192, 8193, 40_960, 60_000], 3000),
                                        ([2049, 4097, 20_000, 95_000], 0),
                                        ([2049, 4097, 20_000, 95_000], 3500)])
@pytest.mark.parametrize("k", [1, 5, 64])
def test_pin_counts_of_huge_nets(oracle_mod, k, sizes, rest):
    n = 100_000
    hgr = nets_around(n, sizes, k, rest)
    part = np.random.default_rng(k).integers(0, max(1, k - 1), size=n).astype(np.int32)
    part[:3] = k - 1  # a block of few pins
    h = create(hgr, 1)
    try:
        d = torch.from_numpy(part).cuda()
        phi, lam = oracle_mod.pin_counts(hgr, k, part)
        got = hg.hg_pin_counts(h, 0, k, d)
        assert np.array_equal(got[0], phi) and np.array_equal(got[1], lam)
        assert np.array_equal(got[2], oracle_mod.block_weights(hgr, k, part))
        assert hg.hg_objective(h, 0, k, d) == oracle_mod.objective(hgr, k, part)
        on = [torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()
              for a in (hgr.offsets, hgr.pins, hgr.net_w, hgr.node_w)]
        assert hg.hg_objective_noalloc(hgr.n, hgr.m, hgr.p, *on, k, d,
                                       torch.cuda.current_stream())[0] == \
            oracle_mod.objective(hgr, k, part)
        if k > 1:
            ref = oracle_mod.lp_refine(hgr, k, part, 50000, 16, 1, 0, 2)
            assert hg.hg_lp_refine(h, 0, k, 50000, 2, d) == (ref["objective"], ref["moves"])
            assert np.array_equal(d.cpu().numpy(), ref["part"])
    finally:
        hg.hg_destroy(h)


# nets around the size above which chunks of a net go to different blocks
@pytest.mark.parametrize("k", [2, 33])
def test_gain_tools_of_huge_nets(oracle_mod, k):
    n = 40_000
    hgr = nets_around(n, [64, 65, 4095, 4096, 4097, 8192, 8193, 32_768, 32_769, 40_000], k)
    rng = np.random.default_rng(k)
    part = rng.integers(0, max(1, k - 1), size=n).astype(np.int32)
    part[:2] = k - 1  # blocks of one or two pins, in different chunks
    nodes = np.concatenate([[0], rng.permutation(np.arange(1, n))[:3000]]).astype(np.int32)
    targets = ((part[nodes] + 1 + rng.integers(0, k - 1, size=len(nodes))) % k).astype(np.int32)
    moved = part.copy()
    moved[nodes] = targets
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()  # noqa: E731
    h = create(hgr, 1)
    try:
        d = dev(part)
        gains = torch.zeros(len(nodes), dtype=torch.int64, device="cuda")
        hg.hg_recalculate_gains(h, 0, k, d, dev(nodes), dev(targets), gains)
        assert np.array_equal(gains.cpu().numpy(),
                              oracle_mod.recalculate_gains(hgr, k, part, nodes, targets))
        b = torch.zeros(n, dtype=torch.int64, device="cuda")
        p = torch.zeros((n, k), dtype=torch.int64, device="cuda")
        hg.hg_gain_table(h, 0, k, d, b, p)
        wb, wp = oracle_mod.gain_table(hgr, k, part)
        assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
        hg.hg_gain_table_move(h, 0, k, d, dev(nodes), dev(targets), b, p)
        wb, wp = oracle_mod.gain_table(hgr, k, moved)
        assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
        assert np.array_equal(d.cpu().numpy(), moved)
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("k", [3, 16, 30, 64])
def test_gain_table_of_hubs(oracle_mod, graph, k):
    """Nodes around the number of nets above which a row is summed by several warps."""
    n, degs = 9000, [511, 512, 513, 1024, 1025, 8000]
    rng = np.random.default_rng(k)
    nets = [[u, int(v)] for u, d in enumerate(degs)
            for v in rng.choice(np.arange(100, n), size=d, replace=False)]
    if not graph:
        nets += [rng.choice(n, size=5, replace=False).tolist() for _ in range(500)]
    hgr = from_nets(n, nets, rng.integers(1, 90_000, size=len(nets)), None)
    part = rng.integers(0, k, size=n).astype(np.int32)
    h = create(hgr, 1)
    try:
        assert hg.hg_level_is_graph(h, 0) == graph
        b = torch.full((n,), 7, dtype=torch.int64, device="cuda")
        p = torch.full((n, k), 7, dtype=torch.int64, device="cuda")
        hg.hg_gain_table(h, 0, k, torch.from_numpy(part).cuda(), b, p)
        wb, wp = oracle_mod.gain_table(hgr, k, part)
        assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
    finally:
        hg.hg_destroy(h)


# candidates on both sides of the twelve parts that a node may have (32-bit ratings:
# nets of 900 pins; 64-bit: of two), above it a table in global memory
@pytest.mark.parametrize("size,count", [(900, 162_000), (900, 163_000), (2, 58_900), (2, 59_200)])
def test_parts_of_a_heavy_node(oracle_mod, size, count):
    n, seed = 200_000, 1
    ids = np.arange(n, dtype=np.uint64)
    hub = int(np.flatnonzero(mix64(ids ^ np.uint64(seed)) % np.uint64(16) == 0)[0])
    rng = np.random.default_rng(size)
    cand = rng.permutation(np.delete(np.arange(n), hub))[:count]
    nets = [[hub, *c.tolist()] for c in np.array_split(cand, -(-count // (size - 1)))]
    nets += [[n - 3, n - 2, n - 1]]
    hgr = from_nets(n, nets, rng.integers(1, 5, size=len(nets)), None)
    ref = oracle_mod.multilevel(hgr, 2, 30000, S=16, factor=160, seed=seed, max_passes=0)
    h = create(hgr, seed)
    try:
        hg.hg_coarsen_level(h, 2)
        assert np.array_equal(hg.hg_get_level(h, 0, with_map=True)["map"], ref.maps[0])
    finally:
        hg.hg_destroy(h)


# one repeated pin in one net: sizes around the classes of the check, many big nets
# in a row
@pytest.mark.parametrize("size", [2, 8, 9, 32, 33, 900, 1024, 1025])
@pytest.mark.parametrize("bad", [None, 0, 299])
def test_repeated_pin_by_net_size(size, bad):
    n, m = 4000, 300
    rng = np.random.default_rng(size)
    pins = np.stack([rng.permutation(n)[:size] for _ in range(m)])
    if bad is not None:
        pins[bad, -1] = pins[bad, 0]
    small = np.stack([rng.permutation(n)[:2] for _ in range(500)])
    off = np.concatenate([[0], size * np.arange(1, m + 1), size * m + 2 * np.arange(1, 501)])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()  # noqa: E731
    args = (n, m + 500, dev(off), dev(np.concatenate([pins.reshape(-1), small.reshape(-1)])), None,
            None, hg.HG_MEM_DEVICE, None, torch.cuda.current_stream())
    if bad is None:
        hg.hg_destroy(hg.hg_create(*args))
    else:
        with pytest.raises(hg.HgError) as ei:
            hg.hg_create(*args)
        assert ei.value.status == hg.HG_ERR_INVALID
