"""Barriers of the single-warp row loops, checked on the CPU.

The loops that advance a stream's full rows (gen_rows_late and gen_rows_short
of the generation kernel, fused_rows and fused_rows_short of the statistics
kernel) read words that other lanes of the warp write, so every read and the
write it must precede or follow need a __syncwarp() between them, also where
one run of rows follows another at once (a request that ends with a row).

This test takes the functions' own source text, compiles it as host code with
traced shared-memory accesses, runs it lane by lane (back-to-back runs of rows
and a row of the general path) and requires that between two barriers no lane
writes a word that another lane reads or writes.  Columns 0 .. N-1 count; the
words behind the row hold nothing that is used.
"""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_07701_gb300", "csrc")

SHIM = r"""
#include <cstdint>
#include <cstdio>
#include <map>
#include <set>
#include <type_traits>
#include <utility>
#define __device__
#define __forceinline__ inline
#define __restrict__
#define MTGP_FULL 0xFFFFFFFFu
static int g_lane, g_epoch;
static uint32_t g_mem[4096];
struct Access { std::set<int> readers, writers; };
static std::map<std::pair<int, uint32_t>, Access> g_log;
static uint32_t rd(uint32_t w) { g_log[{g_epoch, w}].readers.insert(g_lane); return g_mem[w]; }
static void wr(uint32_t w, uint32_t v) { g_log[{g_epoch, w}].writers.insert(g_lane); g_mem[w] = v; }
struct Word {   // one shared word
    uint32_t w;
    operator uint32_t() const { return rd(w); }
    void operator=(uint32_t v) { wr(w, v); }
};
struct Ptr {    // a pointer into the shared row
    uint32_t i;
    Ptr(uint32_t k = 0) : i(k) {}
    Ptr operator+(long k) const { return Ptr((uint32_t)(i + k)); }
    Word operator[](long k) const { return Word{(uint32_t)(i + k)}; }
    Word operator*() const { return Word{i}; }
};
static const uint32_t kS = 0x1000u, kT = 0x100000u;
static uint32_t saddr(Ptr p) { return kS + 4u * p.i; }
static uint32_t saddr(const uint32_t*) { return kT; }
template <int OFF> uint32_t lds_at(uint32_t a)
{
    a += OFF;
    return a >= kT ? 0u : rd((a - kS) / 4u);
}
template <int OFF> void sts_at(uint32_t a, uint32_t v) { wr((a + OFF - kS) / 4u, v); }
static uint32_t __byte_perm(uint32_t x, uint32_t y, uint32_t s)
{
    const uint64_t v = (uint64_t)y << 32 | x;
    uint32_t r = 0;
    for (int i = 0; i < 4; ++i)
        r |= (uint32_t)(v >> 8 * ((s >> 4 * i) & 7) & 255u) << 8 * i;
    return r;
}
static void __syncwarp() { ++g_epoch; }
static uint32_t __ballot_sync(uint32_t, bool) { return 0u; }
static uint32_t __shfl_sync(uint32_t, uint32_t v, uint32_t) { return v; }
static int __ffs(uint32_t x) { return __builtin_ffs((int)x); }
static int __popc(uint32_t x) { return __builtin_popcount(x); }
static void __stcs(uint32_t*, uint32_t) {}
static float __uint_as_float(uint32_t x) { return (float)x; }
static uint32_t __float_as_uint(float x) { return (uint32_t)x; }
template <class F, int... I> void sf(F&& f, std::integer_sequence<int, I...>) { (f(std::integral_constant<int, I>{}), ...); }
template <int N, class F> void static_for(F&& f) { sf(f, std::make_integer_sequence<int, N>{}); }
struct RowP { uint32_t n, mask, pos, sh1, sh2, mirror; };
struct Segment { uint64_t g_start, count, out_off; uint32_t fmt, req; };
struct StatsArgs { uint32_t gmask, hmask, K, t, C; };
struct StatsState { uint32_t lead, D; };
static uint32_t tbl(const uint32_t* t, uint32_t b, uint32_t i) { return t[b + (i & 15u)]; }
static uint32_t temper_index(uint32_t x) { return x; }
static uint32_t temper_pack(const uint32_t (&)[4]) { return 0u; }
template <int FMT> uint32_t finish(uint32_t v, uint32_t) { return v; }
template <int FMT> uint32_t temper_convert(uint32_t v, uint32_t, const uint32_t*) { return v; }
template <class... A> void slow_store(A&&...) {}
static uint32_t hist_addr(const uint32_t*) { return 0u; }
static uint32_t own_addr(const uint32_t*, uint32_t, const StatsArgs&) { return 0u; }
template <class... A> uint32_t gap_run(A&&...) { return 0u; }
template <class... A> uint32_t gap_run_piece(A&&...) { return 0u; }
template <class... A> void gap_window(A&&...) {}
template <class... A> void ham_run(A&&...) {}
template <int KS, class... A> void ham_step(A&&...) {}
template <class... A> void stats_switch(A&&...) {}
static void count_at(uint32_t) {}
"""

MAIN = r"""
static uint32_t g_out[1 << 16], g_tb[64], g_h[64];
static Segment g_seg[1] = {{0u, 1u << 20, 0u, 0u, 0u}};
int main()
{
    const RowP P = {%(n)uu, 0xFFFFFFFFu, %(pos)uu, 3u, 5u, 0u};
    StatsState st{};
    const StatsArgs A = {1u, 1u, 240u, 128u, 4u};
    int epochs = -1;
    for (g_lane = 0; g_lane < 32; ++g_lane) {
        g_epoch = 0;
        const uint32_t lane = (uint32_t)g_lane;
        uint32_t* ow = g_out + 4096;
        Ptr S;
        (void)st; (void)A; (void)ow;
        for (int run = 0; run < 3; ++run) {
            %(rows)s
            if (run == 1) {
                %(part)s
            }
        }
        if (epochs >= 0 && epochs != g_epoch)
            return 2;
        epochs = g_epoch;
    }
    int races = 0;
    for (const auto& kv : g_log) {
        if (kv.first.second >= P.n || kv.second.writers.empty())
            continue;
        std::set<int> all = kv.second.writers;
        all.insert(kv.second.readers.begin(), kv.second.readers.end());
        if (all.size() > 1) {
            if (races++ < 4)
                printf("interval %%d, column %%u: written and touched by %%zu lanes\n", kv.first.first,
                       kv.first.second, all.size());
        }
    }
    printf("races %%d\n", races);
    return 0;
}
"""

# (file, loop, its call, general row path, its call)
LATE = ("mtgp_fast.cuh", "gen_rows_late", "gen_rows_late<%d, 0>(S, ow, P, lane, g_tb, 2u + run);",
        "gen_row_part", "gen_row_part<%d, 0, true>(S, ow, P, lane, g_tb, P.n, 0u, g_seg, 0u, 1u, g_out);")
SHORT = ("mtgp_fast.cuh", "gen_rows_short", "gen_rows_short<%d, 0>(S, ow, P, lane, g_tb, 2u + run);",
         "gen_row_part", "gen_row_part<%d, 0, true>(S, ow, P, lane, g_tb, P.n, 0u, g_seg, 0u, 1u, g_out);")
FUSED = ("mtgp_fused.cuh", "fused_rows",
         "fused_rows<%d, 0, true>(S, ow, P, lane, g_tb, 2u + run, st, g_h, g_h, A);", "fused_row_slow",
         "fused_row_slow<%d>(S, P, lane, g_tb, P.n, 0u, g_seg, 0u, 1u, g_out, st, g_h, g_h, A);")
FSHORT = ("mtgp_fused.cuh", "fused_rows_short",
          "fused_rows_short<%d, 0>(S, ow, P, lane, g_tb, 2u + run, st, g_h, g_h, A);", "fused_row_slow",
          "fused_row_slow<%d>(S, P, lane, g_tb, P.n, 0u, g_seg, 0u, 1u, g_out, st, g_h, g_h, A);")


def _function(text, name):
    """The source of template function `name`, pointers into the shared row
    made traced ones."""
    m = re.search(r"template <[^>]*>\n__device__ __forceinline__ void %s\(" % name, text)
    assert m, name
    i = text.index("{", m.end())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    src = text[m.start():j]
    head, body = src[:i - m.start()], src[i - m.start():]
    assert head.count("uint32_t* S,") == 1
    head = head.replace("uint32_t* S,", "Ptr S,")
    for a, b in (("uint32_t* const Sw = ", "Ptr const Sw = "),
                 ("const uint32_t *Qp[M], *Qq[M];", "Ptr Qp[M], Qq[M];"),
                 ("const uint32_t* const x1_last = ", "Ptr const x1_last = ")):
        body = body.replace(a, b)
    return head + body


def _races(tmp_path, loop, M, n, pos, drop_barrier=False):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    fname, rows, call, part, part_call = loop
    text = open(os.path.join(CSRC, fname)).read()
    fn = _function(text, rows)
    if drop_barrier:   # the one between the loads before the row loop and the loop
        head, tail = fn.split("for (uint32_t q = 0;", 1)
        k = head.rindex("__syncwarp();")
        fn = head[:k] + head[k + len("__syncwarp();"):] + "for (uint32_t q = 0;" + tail
    src = SHIM + fn + "\n" + _function(text, part) + MAIN % {
        "n": n, "pos": pos, "rows": call % M, "part": part_call % M}
    cpp, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    cpp.write_text(src)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-o", str(exe), str(cpp)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout)
    return int(re.search(r"races (\d+)", r.stdout).group(1)), r.stdout


@pytest.mark.parametrize("loop,M,n,pos", [
    (LATE, 11, 351, 95), (LATE, 11, 351, 2), (LATE, 10, 303, 47), (LATE, 23, 726, 470), (LATE, 44, 1391, 1135),
    (SHORT, 4, 101, 37), (SHORT, 4, 101, 2), (SHORT, 5, 133, 69), (SHORT, 4, 128, 64),
    (FUSED, 11, 351, 95), (FUSED, 11, 352, 2), (FUSED, 44, 1391, 1135),
    (FSHORT, 4, 101, 37), (FSHORT, 5, 133, 69)], ids=lambda v: v[1] if isinstance(v, tuple) else str(v))
def test_no_word_is_read_and_written_between_two_barriers(tmp_path, loop, M, n, pos):
    n_races, log = _races(tmp_path, loop, M, n, pos)
    assert n_races == 0, log


@pytest.mark.parametrize("loop,M,n,pos,drop", [
    (LATE, 11, 351, 95, True), (SHORT, 4, 101, 37, True), (FUSED, 11, 351, 95, True), (FSHORT, 4, 101, 37, True),
    (LATE, 11, 351, 96, False), (SHORT, 4, 101, 38, False)], ids=lambda v: v[1] if isinstance(v, tuple) else str(v))
def test_the_check_sees_a_missing_barrier_and_a_short_window(tmp_path, loop, M, n, pos, drop):
    """Controls: without the barrier before the row loop, or one word short
    of the window that the look-ahead needs, the check reports races."""
    assert _races(tmp_path, loop, M, n, pos, drop)[0] > 0
