"""Rules of the kernels' launch code that can be checked without a GPU."""
import glob
import os
import re

from tests import hostcc

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2303_17679_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_cluster_barrier_takes_diverged_warps():
    """barrier.cluster.*.aligned is undefined for a warp whose lanes have not
    rejoined; the phases of the kernels end in loops of per-lane trip counts."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        for ins in re.findall(r'"(barrier\.cluster\.[a-z.]+)', open(path).read()):
            assert ".aligned" not in ins, (os.path.basename(path), ins)
    assert "barrier.cluster.wait.acquire" in source("gridsync.cuh")


def test_buffers_of_a_hook_start_on_a_32_byte_boundary(tmp_path):
    """Whatever alignment the hook's blocks have: the records of k > 32 are read 32
    bytes at a time.  The block itself goes back to the hook."""
    hostcc.run(tmp_path, ["common.cuh"], """
    using namespace hgk;
    void* Alloc::get(size_t bytes) const { return fn_alloc(bytes, ctx); }
    void Alloc::put(void* p) const { fn_free(p, ctx); }
    struct Hook { unsigned char* at; size_t asked; void* freed; };
    int main() {
      std::vector<unsigned char> room(4096);
      for (int shift = 0; shift < 64; ++shift) {
        Hook k{room.data() + shift, 0, nullptr};
        Alloc a;
        a.fn_alloc = [](size_t bytes, void* c) -> void* {
          static_cast<Hook*>(c)->asked = bytes;
          return static_cast<Hook*>(c)->at;
        };
        a.fn_free = [](void* p, void* c) { static_cast<Hook*>(c)->freed = p; };
        a.ctx = &k;
        {
          DBuf<int4> b;
          b.alloc(&a, 10);
          CHECK((uintptr_t)b.p % 32 == 0);
          CHECK((unsigned char*)b.p >= k.at);
          CHECK((unsigned char*)(b.p + 10) <= k.at + k.asked);
          DBuf<int4> c = std::move(b);
          CHECK(!b.p && !k.freed);
        }
        CHECK(k.freed == k.at);
      }
      return 0;
    }
    """)


def test_louvain_vertices_of_any_degree(tmp_path):
    """Every edge of a vertex is covered by its list entries, read at most sixteen
    times, and the entries' numbers stay positive up to the largest degree."""
    hostcc.run(tmp_path, ["louvain.cuh"], """
    using namespace hgk;
    int main() {
      std::vector<long long> degs = {1, 8, 9, 32, 33, 256, 257, 1 << 20, 1 << 26, (1 << 26) + 1,
                                     100000000, (1ll << 31) - 1};
      for (long long d : {4096ll, 32768ll, 33792ll})
        for (long long x = -1; x <= 1; ++x) degs.push_back(d + x);
      int last = 0;
      std::sort(degs.begin(), degs.end());
      for (long long d : degs) {
        int32_t entries = 0;
        if (d > LV_BLOCK) CHECK(lv_class(d, LV_BLOCK, entries) == 5);
        const int cls = lv_class(d, LV_HUGE, entries);
        CHECK(cls >= last && cls < LV_CLASSES && entries >= 1);
        last = cls;
        if (cls < 4) CHECK(entries == 1);
        if (cls == 4) CHECK((long long)entries * LV_PART >= d && entries <= 16);
        if (cls == 5) {
          CHECK((long long)entries * LV_CHUNK >= d && (long long)(entries - 1) * LV_CHUNK < d);
          CHECK(lv_slots(d) >= 2ull * d + 2 && (lv_slots(d) & (lv_slots(d) - 1)) == 0);
        }
      }
      return 0;
    }
    """)


def test_a_wait_lasts_while_the_others_get_on(tmp_path):
    """Blocks may wait for one that sorts tens of millions of moves, so a barrier
    gives up on lack of progress, not after a number of polls."""
    hostcc.run(tmp_path, ["gridsync.cuh"], """
    using namespace hgk;
    int main() {
      WaitBudget still(100);
      int polls = 1;
      while (still.again([] { return 0u; })) ++polls;
      CHECK(polls == 100);
      WaitBudget busy(100);
      unsigned done = 0;
      polls = 0;
      while (polls < 100000 && busy.again([&] { return done; }))
        if (++polls % 90 == 0) ++done;
      CHECK(polls == 100000);
      polls = 0;  // and then it stops
      while (busy.again([&] { return done; })) ++polls;
      CHECK(polls < 200);
      return 0;
    }
    """)


def test_calls_in_flight(tmp_path):
    """Every call counts once, whatever it calls in turn, on its own device."""
    hostcc.run(tmp_path, ["inflight.cuh"], """
    using namespace hgk;
    int main() {
      int a = 0, b = 0, c = 0;
      {
        CallScope outer(0, a);
        CallScope inner(0, a);
        CHECK(calls_in_flight(0) == 1);
        CallScope other(0, b), elsewhere(1, c);
        CHECK(calls_in_flight(0) == 2 && calls_in_flight(1) == 1);
      }
      CHECK(calls_in_flight(0) == 0 && calls_in_flight(1) == 0 && a == 0);
      std::vector<std::thread> t;
      for (int i = 0; i < 8; ++i)
        t.emplace_back([] {
          int depth = 0;
          for (int x = 0; x < 10000; ++x) {
            CallScope s(0, depth);
            if (calls_in_flight(0) < 1) std::abort();
          }
        });
      for (auto& x : t) x.join();
      CHECK(calls_in_flight(0) == 0);
      return 0;
    }
    """)


def test_kernels_of_a_level_are_sized_by_the_calls_in_flight():
    """Not by how a handle waits: plain handles that run at once share the GPU too,
    and one that sleeps alone has all of it."""
    for name in ("cluster.cu", "lp.cu", "community.cu"):
        assert "shares_gpu()" in source(name) and "sync_event" not in source(name), name


def test_kernel_attributes_are_set_by_every_handle(tmp_path):
    """CUDA keeps them per device; a process may hold handles on several."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert "once_flag" not in text, os.path.basename(path)
        if os.path.basename(path) != "common.cuh":
            assert "cudaFuncSetAttribute" not in text, os.path.basename(path)
    hostcc.run(tmp_path, ["common.cuh"], """
    using namespace hgk;
    int main() {
      PreparedKernels one, two;
      int a = 0, b = 0, sets = 0;
      for (int i = 0; i < 3; ++i) {
        one.once(&a, [&] { ++sets; });
        one.once(&b, [&] { ++sets; });
        two.once(&a, [&] { ++sets; });
      }
      CHECK(sets == 3);
      try {
        two.once(&b, [&] { throw 1; });
      } catch (int) {
      }
      two.once(&b, [&] { ++sets; });  // set again after a failure
      CHECK(sets == 4);
      return 0;
    }
    """)


def test_readbacks_go_through_memory_that_no_reset_frees():
    """cudaDeviceReset frees what CUDA allocated on the host; the words of a thread
    outlive handles."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert "cudaHostAlloc" not in text and "cudaMallocHost" not in text, path
    assert "cudaHostRegister" in source("prim.cu")
