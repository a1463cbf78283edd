"""Host-compilable pieces of the library, compiled with g++ and driven here:
what needs no GPU to be shown right."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_14007_gb300", "csrc")


def run_cpp(tmp_path, source):
    """Compiles a C++ program against csrc/ and runs it; its output."""
    gxx = shutil.which("g++") or pytest.skip("no g++")
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(source)
    subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_pair_list_records_store_their_own_entries_only(tmp_path):
    # The records of a chunk are 32 lanes whose stores come in no fixed order:
    # a store outside a record's own places could undo another record's.
    out = run_cpp(tmp_path, r"""
#include <cstdio>
#include "pair_list.h"
int main()
{
    for (uint32_t cnt = 0; cnt <= 15; ++cnt) {
        uint16_t list[32];
        for (uint16_t &x : list) x = 0xABCDu;
        vx::put_nearest_pairs(list + 8, 77u, cnt);
        const uint32_t own = cnt < 4u ? cnt : 4u;
        for (uint32_t i = 0; i < 32; ++i) {
            const bool mine = i >= 8 && i < 8 + own;
            const uint16_t want = mine ? (uint16_t)(77u + ((i - 7u) << 12)) : (uint16_t)0xABCDu;
            if (list[i] != want) return printf("count %u: place %d holds %#x\n", cnt, (int)i - 8, list[i]), 1;
        }
    }
    puts("ok");
}
""")
    assert out.strip() == "ok"


def test_shared_memory_limits_of_two_threads(tmp_path):
    # Two host threads launch the same kernel for the first time, one with
    # much shared memory, one with little: whatever their order, the kernel is
    # allowed as much as the table says.  The large thread's set is held open
    # until the small one has finished (or, kept out meanwhile, for 200 ms).
    out = run_cpp(tmp_path, r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "smem_seen.h"
int main()
{
    static vx::SmemSeen seen;
    std::atomic<size_t> attribute{0};
    std::atomic<bool> large_set{false}, small_done{false};
    std::thread large([&] {
        vx::grow_allowed(seen, 0, 75000, [&](size_t b) {
            attribute = b;
            large_set = true;
            for (int i = 0; i < 200 && !small_done; ++i) std::this_thread::sleep_for(std::chrono::milliseconds(1));
            return 0;
        });
    });
    std::thread small([&] {
        while (!large_set) std::this_thread::yield();
        vx::grow_allowed(seen, 0, 22000, [&](size_t b) { attribute = b; return 0; });
        small_done = true;
    });
    large.join();
    small.join();
    printf("allowed %zu, attribute %zu\n", seen.allowed[0].load(), attribute.load());
    if (seen.allowed[0] != 75000 || attribute != 75000) return 1;
    // a refused size is not remembered, a smaller one needs no call, an
    // unknown device makes the call each time
    int calls = 0;
    if (vx::grow_allowed(seen, 0, 90000, [&](size_t) { return ++calls; }) != 1 || seen.allowed[0] != 75000) return 2;
    if (vx::grow_allowed(seen, 0, 75000, [&](size_t) { return ++calls; }) != 0 || calls != 1) return 3;
    for (int i = 0; i < 2; ++i) vx::grow_allowed(seen, vx::kMaxDevices, 1, [&](size_t) { ++calls; return 0; });
    return calls == 3 ? 0 : 4;
}
""")
    assert out.strip() == "allowed 75000, attribute 75000"


PLANS = r"""
#include <cstdio>
#include "vx_plan.h"
static vx::Plan plan(int K, uint32_t chunks, int part = 0, uint32_t npt = 0, int coarse = -1)
{
    vx_opts o;
    memset(&o, 0, sizeof(o));
    o.size = sizeof(o);
    o.pipeline_chunks = chunks;
    o.partition_log2 = part;
    o.nonces_per_thread = npt;
    o.coarse_bits = coarse;
    vx::Plan p;
    const char *why = nullptr;
    if (vx::make_plan_sized(K, &o, &p, &why, 1024) != VX_OK) p.N = 0;  // refused
    return p;
}
"""


def test_small_partitions_do_not_raise_the_number_of_chunks(tmp_path):
    # Small plots have 4 or 2 times the partitions that 2^11 records would
    # give: a pipelined run still takes no more chunks than with those.
    out = run_cpp(tmp_path, PLANS + r"""
int main()
{
    for (int K = 1; K <= 24; ++K)
        for (uint32_t c : {1u, 2u, 4u, 8u})
            if (plan(K, c).pchunks != plan(K, c, 11).pchunks) return printf("K=%d, %u chunks\n", K, c), 1;
    // where the partition size is the caller's, its partitions count
    if (plan(12, 8, 9).pchunks != 8 || plan(12, 8, 11).pchunks != 2) return 2;
    puts("ok");
}
""")
    assert out.strip() == "ok"


def test_automatic_hash_tiles_follow_the_chunk(tmp_path):
    # A staged hash launch covers one nonce chunk: its automatic nonces per
    # thread are those of the chunk's nonces, and an 11-bit first level comes
    # only with the tile that has a kernel for it.
    out = run_cpp(tmp_path, PLANS + r"""
int main()
{
    for (int K = 1; K <= 32; ++K)
        for (int part : {0, 6, 9, 11})
            for (uint32_t c : {1u, 2u, 4u, 8u}) {
                const vx::Plan p = plan(K, c, part);
                if (p.N == 0) continue;  // refused
                if (p.npt != vx::auto_nonces_per_thread(p.N / p.hchunks) || (p.p1 > 10 && p.npt != 16))
                    return printf("K=%d part %d chunks %d: npt %d, p1 %d\n", K, part, p.hchunks, p.npt, p.p1), 1;
                if (plan(K, c, part, 8).npt != 8 || plan(K, c, part, 16).npt != 16) return 2;
            }
    if (plan(24, 8, 0, 0, 4).npt != 8) return 3;  // two levels of the caller's own, 2^21 nonces a chunk
    puts("ok");
}
""")
    assert out.strip() == "ok"


def test_the_untuned_plan_is_a_tuning_candidate(tmp_path):
    # Whatever the planner picks by itself is among the plans the autotuner
    # times, so a tuned plot is not slower than an untuned one.
    out = run_cpp(tmp_path, PLANS + r"""
int main()
{
    int plans = 0;
    for (int K = 1; K <= 32; ++K)
        for (uint32_t chunks : {0u, 2u, 8u})
            for (uint32_t fuse : {0u, 1u})
                for (uint32_t win : {0u, 2u})
                    for (uint32_t place : {0u, 1u}) {
                        vx_opts base;
                        memset(&base, 0, sizeof(base));
                        base.size = sizeof(base);
                        base.coarse_bits = -1;
                        base.pipeline_chunks = chunks;
                        base.fuse_pair_hash = fuse;
                        base.window_bits = win;
                        base.t2_placement = place;
                        vx::Plan own, p;
                        const char *why = nullptr;
                        if (vx::make_plan_sized(K, &base, &own, &why, 1024) != VX_OK) continue;
                        bool found = false;
                        for (const vx_opts &o : vx::tune_candidates(base))
                            found = found || (vx::make_plan_sized(K, &o, &p, &why, 1024) == VX_OK && vx::same_plan(own, p));
                        if (!found) return printf("K=%d chunks %u fuse %u window_bits %u\n", K, chunks, fuse, win), 1;
                        ++plans;
                    }
    puts(plans > 300 ? "ok" : "few plans");
}
""")
    assert out.strip() == "ok"
