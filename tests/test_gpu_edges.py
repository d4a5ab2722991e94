"""The edges of the kernels' size classes on the GPU against the oracle: net sizes
around every class of the grouped pins, the contraction, the cluster refresh and
the gain tools, block counts around the label propagation's kernels, and levels
on both sides of the bitmap and one-launch limits.  All results are integers and
every comparison is exact."""
import numpy as np
import pytest

import synth
from tests.tiny import from_nets

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2303_17679_gb300 import hg  # noqa: E402

SIZES = [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 511, 512, 513,
         1023, 1024, 1025, 2048, 2049]
HUGE = [4095, 4096, 4097, 9000]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def edge_nets(n, sizes, repeat, seed, span=None, hub=0):
    """`repeat` nets of every size with pins among the first `span` nodes (every
    third one a copy of the net before it), and `hub` pairs at node 0."""
    rng = np.random.default_rng(seed)
    span = min(n, span or n)
    nets = []
    for size in sizes:
        for r in range(repeat if size <= 64 else max(3, repeat // 8)):
            if r % 3 == 2:
                nets.append(rng.permutation(nets[-1]).tolist())
            else:
                nets.append(rng.choice(span, size=min(size, span), replace=False).tolist())
    nets += [[0, int(v)] for v in rng.choice(np.arange(1, span), size=hub)]
    order = rng.permutation(len(nets))
    return from_nets(n, [nets[i] for i in order], rng.integers(1, 9, size=len(nets)),
                     rng.integers(1, 4, size=n))


def create(hgr, seed, S=16, T=1000, factor=160, communities=0):
    o = hg.hg_default_options()
    o.seed, o.subrounds, o.rating_max_net_size = seed, S, T
    o.contraction_limit_factor, o.community_detection = factor, communities
    return hg.hg_create(hgr.n, hgr.m, hgr.offsets, hgr.pins, hgr.net_w, hgr.node_w,
                        hg.HG_MEM_HOST, o, torch.cuda.current_stream())


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.int32)).cuda()


# S = 1: every node decides at once, so a net sees more joins than its set holds.
# T above 1024: rated nets of every refresh class.  n, span: coarse nodes below and
# above the limits of the bitmap forms.
@pytest.mark.parametrize("n,sizes,span,S,T,repeat,hub", [
    (3000, SIZES + HUGE, 3000, 1, 1000, 60, 0),
    (3000, SIZES, 3000, 16, 1024, 30, 400),
    (6000, [2, 33, 1024, 1025, 2049, 4097], 6000, 5, 5000, 16, 900),
    (60_000, SIZES + HUGE, 60_000, 16, 64, 300, 9000),
    (700_000, SIZES + HUGE, 100_000, 16, 300, 60, 300)])
def test_coarsening_at_the_edges(oracle_mod, n, sizes, span, S, T, repeat, hub):
    hgr = edge_nets(n, sizes, repeat, n + S, span, hub)
    seed, k = 5, 2
    vc = oracle_mod.multilevel(hgr, k, S=S, T=T, factor=20, seed=seed, max_passes=0)
    h = create(hgr, seed, S, T, 20)
    try:
        while hg.hg_coarsen_level(h, k)[0] == hg.HG_OK:
            pass
        assert hg.hg_num_levels(h) == len(vc.levels) and len(vc.levels) > 1
        for lv in range(1, len(vc.levels)):
            assert np.array_equal(hg.hg_get_level(h, lv - 1, with_map=True)["map"],
                                  vc.maps[lv - 1])
            got, want = hg.hg_get_level(h, lv), vc.levels[lv]
            assert np.array_equal(got["offsets"], want.offsets)
            assert np.array_equal(got["pins"], want.pins)
            assert np.array_equal(got["net_w"], want.net_w)
            assert np.array_equal(got["node_w"], want.node_w)
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("n,m,span,S", [(2000, 9000, 200, 16), (50_000, 60_000, 50_000, 3)])
def test_graph_contraction_at_the_edges(oracle_mod, n, m, span, S):
    """Parallel edges, edges inside a cluster, isolated nodes."""
    rng = np.random.default_rng(n)
    a = rng.integers(0, span, size=m)
    b = (a + 1 + rng.integers(0, min(span - 1, 40), size=m)) % span
    hgr = from_nets(n, np.stack([a, b], 1).tolist(), rng.integers(1, 50, size=m),
                    rng.integers(1, 4, size=n))
    vc = oracle_mod.multilevel(hgr, 2, S=S, factor=10, seed=3, max_passes=2)
    h = create(hgr, 3, S, factor=10)
    try:
        assert hg.hg_level_is_graph(h, 0)
        part = torch.empty(n, dtype=torch.int32, device="cuda")
        obj = hg.hg_partition(h, 2, 30000, 2, part)
        assert hg.hg_num_levels(h) == len(vc.levels)
        for lv in range(1, len(vc.levels)):
            got, want = hg.hg_get_level(h, lv), vc.levels[lv]
            assert np.array_equal(got["pins"], want.pins)
            assert np.array_equal(got["net_w"], want.net_w)
        assert np.array_equal(part.cpu().numpy(), vc.parts[0]) and obj == vc.objectives[0]
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("k", [2, 8, 9, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("n,repeat,hub", [(3000, 30, 700), (40_000, 600, 20_000)])
def test_label_propagation_at_the_edges(oracle_mod, k, n, repeat, hub):
    """hub: a node whose nets are split over several items."""
    hgr = edge_nets(n, SIZES + (HUGE if n > 9000 else []), repeat, n + k, hub=hub)
    part0 = np.random.default_rng(k).integers(0, k, size=n).astype(np.int32)
    ref = oracle_mod.lp_refine(hgr, k, part0, 50000, 16, 4, 0, 3)
    h = create(hgr, 4)
    try:
        d = dev(part0)
        obj, moves = hg.hg_lp_refine(h, 0, k, 50000, 3, d)
        assert np.array_equal(d.cpu().numpy(), ref["part"])
        assert (obj, moves) == (ref["objective"], ref["moves"])
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("k,frac", [(2, 0.5), (7, 0.02), (33, 1.0), (64, 0.3)])
def test_gain_tools_at_the_edges(oracle_mod, k, frac):
    hgr = edge_nets(12_000, SIZES + HUGE, 60, k, hub=5000)
    rng = np.random.default_rng(k)
    part = rng.integers(0, k, size=hgr.n).astype(np.int32)
    nodes = rng.permutation(hgr.n)[: int(frac * hgr.n)].astype(np.int32)
    targets = ((part[nodes] + 1 + rng.integers(0, k - 1, size=len(nodes))) % k).astype(np.int32)
    moved = part.copy()
    moved[nodes] = targets
    h = create(hgr, 1)
    try:
        d = dev(part)
        gains = torch.zeros(len(nodes), dtype=torch.int64, device="cuda")
        hg.hg_recalculate_gains(h, 0, k, d, dev(nodes), dev(targets), gains)
        assert np.array_equal(gains.cpu().numpy(),
                              oracle_mod.recalculate_gains(hgr, k, part, nodes, targets))
        b = torch.zeros(hgr.n, dtype=torch.int64, device="cuda")
        p = torch.zeros((hgr.n, k), dtype=torch.int64, device="cuda")
        hg.hg_gain_table(h, 0, k, d, b, p)
        hg.hg_gain_table_move(h, 0, k, d, dev(nodes), dev(targets), b, p)
        wb, wp = oracle_mod.gain_table(hgr, k, moved)
        assert np.array_equal(b.cpu().numpy(), wb) and np.array_equal(p.cpu().numpy(), wp)
        assert np.array_equal(d.cpu().numpy(), moved)
        assert hg.hg_objective(h, 0, k, d) == oracle_mod.objective(hgr, k, moved)
    finally:
        hg.hg_destroy(h)
    obj, bw = hg.hg_objective_noalloc(hgr.n, hgr.m, hgr.p, dev(hgr.offsets), dev(hgr.pins),
                                      dev(hgr.net_w), dev(hgr.node_w), k, dev(moved),
                                      torch.cuda.current_stream())
    assert obj == oracle_mod.objective(hgr, k, moved)
    assert np.array_equal(bw, oracle_mod.block_weights(hgr, k, moved))


# both sides of the one-launch limit (8192 nodes) and of the packed weights (2^20)
@pytest.mark.parametrize("n", [1, 31, 33, 8192, 8193, 30_000])
@pytest.mark.parametrize("k,heavy", [(1, 1), (2, 1 << 20), (33, (1 << 20) + 1), (64, 7),
                                     (64, 1 << 26)])
def test_initial_partition_at_the_edges(oracle_mod, n, k, heavy):
    rng = np.random.default_rng(n + k)
    c = rng.integers(1, 5, size=n).astype(np.int32)
    c[rng.integers(0, n, size=4)] = heavy
    hgr = from_nets(n, [[0, n - 1]] if n > 1 else [], None, c)
    h = create(hgr, 9)
    try:
        part = torch.empty(n, dtype=torch.int32, device="cuda")
        hg.hg_initial_partition(h, 0, k, part)
        assert np.array_equal(part.cpu().numpy(), oracle_mod.initial_partition(c, k, 9))
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("n,hub", [(3000, 300), (20_000, 15_000)])
def test_communities_at_the_edges(oracle_mod, n, hub):
    """Vertices of more than 32, 256 and 4096 neighbours on both sides."""
    hgr = edge_nets(n, SIZES + (HUGE if n > 9000 else []), 30, n, hub=hub)
    want, levels, moves = oracle_mod.communities(hgr, S=16, seed=2)
    h = create(hgr, 2)
    try:
        hg.hg_detect_communities(h)
        assert np.array_equal(hg.hg_get_communities(h, 0), want)
        st = hg.hg_get_stats(h)
        assert st["louvain_levels"] == levels and st["louvain_moves"] == moves
    finally:
        hg.hg_destroy(h)


@pytest.mark.parametrize("bad", [None, 0, 699])
def test_repeated_pin_among_many_big_nets(bad):
    n, m, size = 5000, 700, 1100
    rng = np.random.default_rng(1)
    pins = np.concatenate([rng.permutation(n)[:size] for _ in range(m)]).astype(np.int32)
    if bad is not None:
        pins[bad * size + size - 1] = pins[bad * size]
    off = np.arange(m + 1, dtype=np.int32) * size
    args = (n, m, dev(off), dev(pins), dev(np.ones(m)), dev(np.ones(n)), hg.HG_MEM_DEVICE, None,
            torch.cuda.current_stream())
    if bad is None:
        hg.hg_destroy(hg.hg_create(*args))
    else:
        with pytest.raises(hg.HgError) as ei:
            hg.hg_create(*args)
        assert ei.value.status == hg.HG_ERR_INVALID
