"""The library's host-side choices (csrc/kvd_rules.cpp), compiled alone with the
host compiler: no GPU, no library.  The device's part of them, how many clusters
of a shape it holds at once, is a table of what a GB300 answers."""
import ctypes
import os
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_12707_gb300", "csrc")


def compile_host(path, source, *files):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    src, lib = os.path.join(path, "shim.cpp"), os.path.join(path, "shim.so")
    with open(src, "w") as f:
        f.write(textwrap.dedent(source))
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    src, *(os.path.join(CSRC, x) for x in files), "-o", lib], check=True)
    return ctypes.CDLL(lib)


#: clusters of (CTAs, warps) with 1, 2, .. ring stages that a GB300 holds at once, by head_dim
RESIDENT = {
    128: {(8, 8): (15, 15, 15), (8, 4): (51, 51, 36), (4, 4): (110, 110, 74), (2, 4): (228, 228, 152),
          (1, 4): (456, 456, 304)},
    64: {(8, 8): (36, 36, 36, 15, 15, 15), (8, 4): (74, 74, 74, 51, 36, 36), (4, 4): (148, 148, 148, 110, 74, 74),
         (2, 4): (304, 304, 304, 228, 152, 152), (1, 4): (608, 608, 608, 456, 304, 304)},
}
WARPS = 152 * 8   # resident warps of the split pass


class Rules:
    def __init__(self, lib):
        self.lib = lib
        for d, shapes in RESIDENT.items():
            for (c, w), counts in shapes.items():
                for r, n in enumerate(counts):
                    lib.set_resident(d, c, w, r + 1, n)

    def shape(self, hq, hkv, d, pages, spread=False, limit=0):
        """(CTAs, warps, stages) of a step over rows of these page counts; no CTAs: a split plan."""
        out = (ctypes.c_int * 3)()
        self.lib.shape(d, int(hq > hkv), hkv, len(pages), sum(pages), max(pages), int(spread), limit, out)
        return tuple(out)


    def item_pages(self, hq, hkv, d, pages, growing=False):
        return self.lib.item_pages(d, int(hq > hkv), hkv, WARPS, len(pages), sum(pages), max(pages), int(growing))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    return Rules(compile_host(str(tmp_path_factory.mktemp("rules")), """
        #include "kvd_internal.h"
        using namespace kvd;
        static int known[2][9][9][8];
        static int resident(int, int D, bool, const ClusterShape& s) { return known[D == 128][s.ctas][s.warps][s.ring]; }
        extern "C" void set_resident(int D, int c, int w, int r, int n) { known[D == 128][c][w][r] = n; }
        extern "C" void shape(int D, int gqa, int hkv, int rows, int pages, int max_pages, int spread, int limit,
                              int* out)
        {
            const ClusterShape s = pick_cluster_shape(resident, 0, D, gqa, hkv, rows, pages, max_pages, spread, limit);
            out[0] = s.ctas;
            out[1] = s.warps;
            out[2] = s.ring;
        }
        extern "C" int item_pages(int D, int gqa, int hkv, int warps, int rows, int pages, int max_pages, int growing)
        {
            return auto_item_pages(D, gqa, hkv, warps, rows, pages, max_pages, growing);
        }
        extern "C" int whole(int D, int group, int hkv, int rows, int pages, int max_pages)
        {
            return whole_rows_beat_clusters(D, group, hkv, rows, pages, max_pages);
        }
        extern "C" int noalloc_cap(int gqa, int hkv, int warps, int rows, int pages, int max_pages, int T)
        {
            return noalloc_chunk_cap(gqa, hkv, warps, rows, pages, max_pages, T);
        }
        extern "C" int step_launch(int rows, int64_t ids, int* threads)
        {
            *threads = step_threads(rows, ids);
            return step_ctas(rows, ids);
        }
        extern "C" int early(int ctas, int slots) { return place_first_layer_early(ctas, slots); }
        extern "C" int cap(int gqa, int units, int warps, int max_pages, int T)
        {
            return chunk_cap(gqa, units, warps, max_pages, T);
        }
    """, "kvd_rules.cpp"))


def pages_of(lens):
    return [(n + 15) // 16 for n in lens]


@pytest.mark.parametrize("Hq,Hkv,d,lens,shape", [   # the steps of the GPU test of every cluster shape, after one token
    (28, 4, 128, [2200, 33], (8, 8)),
    (14, 2, 64, [2300, 0], (8, 8)),
    (8, 8, 128, [700, 1, 16, 15], (8, 4)),
    (56, 8, 128, [300, 511, 512], (8, 4)),
    (16, 16, 128, [300, 17, 0, 31, 250], (4, 4)),
    (24, 24, 64, [100, 64, 63, 1, 47], (2, 4)),
    (16, 8, 128, [90, 0, 15, 16, 47, 90, 3, 2, 77, 61, 33, 32], (2, 4)),
    (8, 8, 64, [60 - 3 * (b % 20) for b in range(24)], (1, 4)),
    (6, 2, 64, [40 - (b % 40) for b in range(120)], (1, 4)),
])
def test_cluster_shapes_of_small_steps(rules, Hq, Hkv, d, lens, shape):
    assert rules.shape(Hq, Hkv, d, pages_of([n + 1 for n in lens]))[:2] == shape


@pytest.mark.parametrize("growing", [False, True])
@pytest.mark.parametrize("Hq,Hkv,d,pages", [
    (32, 32, 128, [229]),
    (32, 32, 128, [91, 88, 85]),
    (8, 8, 128, [263, 257, 250]),
    (56, 8, 128, [571, 560, 541]),
    (56, 8, 128, [774, 760, 742]),
    (8, 8, 64, [738] * 3),
    (14, 2, 128, [399 + 2 * b for b in range(17)]),
])
def test_one_item_per_warp_is_not_a_few_more(rules, Hq, Hkv, d, pages, growing):
    """Even rows of short shares get one item per resident warp: with a few
    more, some warps would work a second one while all others wait."""
    T = rules.item_pages(Hq, Hkv, d, pages, growing)
    items = sum(-(-n // T) for n in pages) * Hkv
    assert 0.75 * WARPS <= items <= WARPS


@pytest.mark.parametrize("growing", [False, True])
@pytest.mark.parametrize("Hq,Hkv,d,pages", [
    (32, 32, 128, [1001]),
    (32, 32, 128, [501] * 2),
    (40, 40, 128, [404] * 2),
    (32, 32, 128, [200, 195, 190]),
    (14, 2, 64, [1873 - 11 * b for b in range(13)]),
])
def test_long_shares_of_few_units_have_several_items_per_warp(rules, Hq, Hkv, d, pages, growing):
    T = rules.item_pages(Hq, Hkv, d, pages, growing)
    assert T <= -(-sum(pages) * Hkv // ((2 if Hq > Hkv else 3) * WARPS))


@pytest.mark.parametrize("Hq,Hkv,d,pages,whole", [
    (40, 40, 128, [7] + [1 + b % 2 for b in range(10)], (False, False)),
    (8, 8, 128, [8] + [2 + b % 2 for b in range(32)], (False, False)),
    (32, 32, 128, [7] + [1 + b % 3 for b in range(20)], (False, False)),
    (8, 8, 128, [6] + [2 + b % 3 for b in range(98)], (True, False)),
    (40, 40, 128, [7] + [2 + b % 3 for b in range(33)], (True, True)),
    (16, 8, 128, [4] + [1] * 27, (True, False)),
    (28, 4, 128, [5] + [2] * 60, (True, False)),
])
def test_short_unequal_rows_stay_whole_only_where_it_pays(rules, Hq, Hkv, d, pages, whole):
    """A long row kept whole is one warp's work while the others wait; device
    steps launch the merge pass in any case."""
    assert tuple(rules.item_pages(Hq, Hkv, d, pages, growing) >= max(pages) for growing in (False, True)) == whole


@pytest.mark.parametrize("d,group,hkv,pages,whole", [
    (128, 7, 4, [1] * 51, True),
    (128, 1, 32, [1], True),
    (64, 7, 2, [1, 1], True),
    (64, 3, 2, [1, 1], False),
    (64, 7, 2, [1] * 111, True),
    (128, 7, 4, [2, 1, 2], True),
    (128, 2, 8, [2] + [1] * 42, True),
    (128, 1, 40, [2], False),
    (64, 7, 2, [2, 1] * 38, False),
    (128, 7, 2, [3] + [1] * 60, False),
])
def test_rows_of_one_or_two_pages_stay_whole(rules, d, group, hkv, pages, whole):
    assert bool(rules.lib.whole(d, group, hkv, len(pages), sum(pages), max(pages))) == whole


@pytest.mark.parametrize("Hq,Hkv,d,lens,clusters", [
    (8, 8, 128, [3953, 3162], False),
    (8, 8, 128, [2330, 1500, 800, 200, 150, 100], False),
    (40, 40, 128, [380, 190, 100, 60, 40, 30, 20, 15, 10], False),
    (32, 32, 128, [290, 29, 40, 50, 60, 30, 35, 45, 70], False),
    (8, 8, 64, [9200, 1500], False),
    (8, 8, 64, [795] + [19 + b * 4 for b in range(28)], False),
    (16, 16, 128, [5000], False),
    (32, 32, 128, [2000], True),
    (32, 32, 128, [900, 500, 300], True),
    (40, 40, 128, [730, 400, 80], True),
    (8, 8, 128, [7000], True),
    (8, 8, 64, [1080 - 40 * b for b in range(17)], True),
    (28, 4, 128, [4000, 2500], True),
])
def test_clusters_where_the_longest_rows_warps_keep_up(rules, Hq, Hkv, d, lens, clusters):
    assert (rules.shape(Hq, Hkv, d, pages_of(lens))[0] > 0) == clusters


def test_small_grids_are_not_placed_beside_the_step_kernel(rules):
    assert not any(rules.lib.early(n, WARPS) for n in (1, 256, 512, 607))
    assert all(rules.lib.early(n, WARPS) for n in (608, 1216))


@pytest.mark.parametrize("Hq,Hkv,d,B", [(32, 32, 128, 1), (28, 4, 128, 8), (8, 8, 64, 4), (14, 2, 64, 13), (32, 32, 128, 12)])
def test_rows_that_start_short_fill_the_gpu_when_grown(rules, Hq, Hkv, d, B):
    """Device steps keep the target size of the lengths held when they were
    enabled: few units of a page each still get as many items as 60 grown
    pages make, up to three per warp or the cap."""
    for held in (1, 2, 4):
        T = rules.item_pages(Hq, Hkv, d, [held] * B, True)
        items = min(-(-60 // T), rules.lib.cap(int(Hq > Hkv), B * Hkv, WARPS, 256, T)) * B * Hkv
        assert items >= min(WARPS, 30 * B * Hkv, 16 * B * Hkv if Hq > Hkv else WARPS)
@pytest.mark.parametrize("Hq,Hkv,d,B", [(32, 32, 128, 1), (28, 4, 128, 1), (28, 4, 128, 4), (28, 4, 128, 8), (40, 40, 128, 1),
                                        (8, 8, 64, 4), (14, 2, 64, 8), (32, 32, 128, 3), (8, 8, 128, 4), (6, 2, 64, 60)])
@pytest.mark.parametrize("limit", [20, 64, 200, 256, 512, 2048, 8192])
def test_a_shape_that_stays_serves_grown_rows(rules, Hq, Hkv, d, B, limit):
    """Device steps keep the clusters they started with (a captured graph
    does), so those picked for a page a row have the warps, and the stages,
    that rows of `limit` pages need; else the step runs from a plan."""
    for held in (1, 4, 10):
        c, w, r = rules.shape(Hq, Hkv, d, [held] * B, limit=limit)
        if c == 0:
            continue
        n = c * w
        if limit > 2 * n:
            assert r >= 2
        items = 64 if B * Hkv * 32 < WARPS else 16 if Hq > Hkv else 32   # of the plan, for one long row
        assert -(-limit // n) <= max(18, -(-limit // items)) or (B == 1 and Hkv * n > 900)
    assert rules.shape(Hq, Hkv, d, [10] * B, limit=11) == rules.shape(Hq, Hkv, d, [10] * B)


def test_clusters_of_long_tables(rules):
    assert rules.shape(32, 32, 128, [4], limit=256) == (8, 4, 3)     # one request in a 4096-token context
    assert rules.shape(28, 4, 128, [4] * 2, limit=2048) == (8, 8, 3)
    assert rules.shape(28, 4, 128, [4] * 8, limit=512) == (8, 4, 3)
    assert rules.shape(28, 4, 128, [4] * 8, limit=520) == (8, 4, 3)  # 8192 tokens and a little room
    assert rules.shape(28, 4, 128, [4] * 8, limit=2048) == (0, 0, 0)
    assert rules.shape(32, 32, 128, [4] * 3, limit=256) == (0, 0, 0)


def test_few_units_get_the_items_that_their_rows_ask_for(rules):
    """Units that would leave resident warps without an item at the usual cap
    are cut into items of T pages, not fewer larger ones."""
    for gqa in (0, 1):
        for units in (1, 8, 32, 37):
            for T in (2, 7, 14):
                for pages in (1, 16 * T, 16 * T + 1, 31 * T, 32 * T, 33 * T, 64 * T):
                    assert rules.lib.cap(gqa, units, WARPS, pages, T) >= min(64, -(-pages // T))
    assert rules.lib.cap(1, 38, WARPS, 2000, 2) == 16 and rules.lib.cap(0, 38, WARPS, 2000, 2) == 32


@pytest.mark.parametrize("Hq,Hkv,pages,cap", [
    (28, 4, [1347] + [337] * 12, 32),
    (16, 8, [1786, 1500, 900, 600, 400, 228], 32),
    (14, 2, [721] + [18] * 25, 32),
    (28, 4, [288, 270, 260, 160, 150, 140] + [60] * 26, 16),
    (28, 4, [300] * 20, 16),
    (8, 8, [721] + [18] * 70, 32),
])
def test_the_allocation_free_call_cuts_a_long_row_into_32(rules, Hq, Hkv, pages, cap):
    assert rules.lib.noalloc_cap(int(Hq > Hkv), Hkv, WARPS, len(pages), sum(pages), max(pages), 8) == cap


def test_step_kernels_have_warps_for_their_rows(rules):
    """Many short rows need warps as many long ones do; a row needs a thread of
    its own unless the block has 1024."""
    def launch(rows, ids):
        t = ctypes.c_int()
        return rules.lib.step_launch(rows, ctypes.c_int64(ids), ctypes.byref(t)), t.value

    for rows in (1, 8, 9, 16, 17, 64, 65, 141, 188, 256, 257, 512, 513, 1024, 3000):
        for per_row in (0, 1, 3, 60, 2049):
            c, t = launch(rows, rows * per_row)
            assert t in (256, 512, 1024) and c in (1, 8) and (t >= rows or t == 1024)
            if per_row == 0:
                assert c == 1
            else:
                assert c * t // 32 >= min(rows, 128) // 2
    assert launch(12, 12 * 128) == launch(12, 12 * 2048)
    assert launch(188, 188)[0] == 8


def test_setup_runs_once_on_each_device(tmp_path):
    """A kernel attribute holds on the device it was set on: the second device
    gets its own call, a failed one is tried again."""
    lib = compile_host(str(tmp_path), """
        #include "kvd_internal.h"
        static kvd::OncePerDevice once;
        static int calls[128];
        extern "C" int setup(int device, int result)
        {
            return once(device, [&] { ++calls[device]; return (cudaError_t)result; });
        }
        extern "C" int count(int device) { return calls[device]; }
    """)
    assert [lib.setup(0, 0), lib.setup(0, 0), lib.setup(1, 0), lib.setup(0, 0), lib.setup(1, 0)] == [0] * 5
    assert [lib.count(0), lib.count(1)] == [1, 1]
    assert [lib.setup(2, 1), lib.setup(2, 0), lib.setup(2, 1)] == [1, 0, 0] and lib.count(2) == 2
    assert [lib.setup(100, 0), lib.setup(100, 0)] == [0, 0] and lib.count(100) == 2   # past the table: every time
