// Register-resident MTGP32 generation kernel for sm_103a.
//
// Streams are advanced by one warp each (the paper's "PRNG per block of
// threads", Sec. 2, with the state on chip while it is advanced and in global
// memory between launches), or -- for the longest streams of a launch -- by
// all G warps of a CTA together.
//
// Layout of a stream's state while it is on chip:
//   * The sequence is cut into rows of N words: column c of row q holds
//     x_{qN + c}.  Computing row q+1 column c needs (row q, c) and
//     (row q, c+1) [the words i and i+1 of the recurrence] and the word i+pos,
//     which is (row q, c+pos) when c+pos < N and (row q+1, c+pos-N) otherwise;
//     the tempering word i+pos-1 likewise.  So a state needs only the latest
//     value of each column.
//   * Column group m (columns 32m .. 32m+31) belongs to one warp; lane l of
//     that warp keeps column 32m + l in a register (word i).
//   * The latest value of every column is also published in a shared-memory
//     row S[0..N), where words i+1 and i+pos of 32 consecutive columns are
//     plain conflict-free loads.  A pick-up past column N-1 is the new row's
//     value of column c+pos-N: the late-tempering loops keep each group's
//     pick-up address with that wrap in it; the other loops (CTA-wide
//     streams, K = 8, N - pos < 256) mirror columns 0..E-1, E >= pos + 31,
//     at S[N..N+E), so that S[c+1], S[c+pos] and S[c+pos-1] need no wrap.
//   * The recursion and tempering tables are 16-word shared arrays whose entry
//     k sits in bank k, so a warp's 32 lookups are one conflict-free
//     shared-memory wavefront whatever the indices.
//
// A sub-step m computes columns 32m..32m+31 of the next row (one new word per
// lane).  K consecutive sub-steps form one parallel step of 32K words; when
// 32K <= N - pos none of them reads a word produced in the same step (the
// block-parallel window of the method), so a step reads everything, passes a
// barrier, then writes everything.
#pragma once

#include <utility>

#include "mtgp_internal.h"

namespace mtgp {

#define MTGP_FULL 0xFFFFFFFFu

__device__ __forceinline__ void cp_async16(uint32_t* smem_dst, const uint32_t* gsrc)
{
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gsrc) : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t sm_id()
{
    uint32_t v;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(v));
    return v;
}

// Timeline record of one item (only when a trace buffer is given).
__device__ __forceinline__ void trace_item(uint64_t* trace, uint32_t it, uint64_t t0,
                                           const Segment* segs, const WorkItem& w)
{
    const Segment last = segs[w.seg_begin + w.nseg - 1u];
    trace[4u * it + 0] = t0;
    trace[4u * it + 1] = global_ns();
    trace[4u * it + 2] = sm_id();
    trace[4u * it + 3] = last.g_start + last.count;
}

__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Per-stream scalars the row code reads: the handle's parameter set, or the
// stream's own set when the handle has one per stream (all sets of a handle
// share N and the mask).  Kept in registers for the whole item.
struct RowP {
    uint32_t n, mask, pos, sh1, sh2, mirror;
};

// Tables in shared memory: 16 words each, at a 64-byte aligned base, so
// that entry k of a table sits in bank k and any lookup pattern of a warp is
// one conflict-free wavefront.  Tb[0..16) recursion, Tb[16..32) tempering,
// Tb[32..48) float tempering.
__device__ __forceinline__ uint32_t tbl(const uint32_t* Tb, uint32_t base, uint32_t idx)
{
    return Tb[base + (idx & 15u)];
}

// Tempering index from word i+pos-1: fold >> 16 then >> 8; the low four bits
// select the entry.
__device__ __forceinline__ uint32_t temper_index(uint32_t xq)
{
    const uint32_t t = xq ^ (xq >> 16);
    return t ^ (t >> 8);
}

// Output conversion from the new word v and the tempering index ti.
//   FMT 0: v ^ TMP[ti]
//   FMT 1: (v >> 9) ^ FLT[ti]   == 0x3F800000 | ((v ^ TMP[ti]) >> 9)
//   FMT 2: the FMT 1 float minus 1.0f (exact: Sterbenz)
template <int FMT>
__device__ __forceinline__ uint32_t temper_convert(uint32_t v, uint32_t ti, const uint32_t* Tb)
{
    if (FMT == 0)
        return v ^ tbl(Tb, 16u, ti);
    const uint32_t b = (v >> 9) ^ tbl(Tb, 32u, ti);
    if (FMT == 1)
        return b;
    return __float_as_uint(__uint_as_float(b) - 1.0f);
}

// Per-lane output of the slow path: the lane finds its request and format
// (ou / of are the u32 and [1,2) outputs).
__device__ __forceinline__ void slow_store(uint32_t ou, uint32_t of, uint64_t g,
                                           const Segment* __restrict__ segs, uint32_t s_first,
                                           uint32_t s_end, uint32_t* __restrict__ out)
{
    uint32_t s = s_first;
    while (s + 1 < s_end && g >= segs[s + 1].g_start)
        ++s;
    const Segment sg = segs[s];
    uint32_t o = ou;
    if (sg.fmt == 1)
        o = of;
    else if (sg.fmt == 2)
        o = __float_as_uint(__uint_as_float(of) - 1.0f);
    out[sg.out_off + (g - sg.g_start)] = o;
}

// ===========================================================================
// Rows.  A row is "full" when all N of its words go to one request; other
// rows (the last, partial row of a stream, or a row crossing requests) take
// the slow path where each lane finds its own request.
//
// Work split: sub-step m of a row belongs to warp (m mod WG) of the WG warps
// advancing the stream (WG = 1 for a warp-owned stream); that warp keeps
// columns 32m + lane in register r[m / WG].  `Sw` = S + 32*warp + lane.
//
// No warp-synchronous instruction is executed under a lane-dependent
// condition: the write phase is lane-predicated and holds only stores.
//
// S, Sw and Q all point into the same shared row (and ow into `out`), so
// none of them is __restrict__: the loads of one step must stay after the
// stores of the previous one.
// ===========================================================================
template <int M, int K, int WG, int FMT, bool SLOW>
__device__ __forceinline__ void gen_row(uint32_t (&r)[(M + WG - 1) / WG], uint32_t* S,
                                        uint32_t* Sw, uint32_t* ow,
                                        const uint32_t* Q, const RowP& P,
                                        uint32_t warp, uint32_t lane, const uint32_t* __restrict__ Tb,
                                        uint32_t last_lane, uint32_t n_valid, uint64_t row_g,
                                        const Segment* __restrict__ segs, uint32_t s_first,
                                        uint32_t s_end, uint32_t* __restrict__ out)
{
    constexpr int J = (M + WG - 1) / WG;
    constexpr int PER = K / WG;   // sub-steps per warp in one parallel step
#pragma unroll
    for (int s0 = 0; s0 < M; s0 += K) {
        if (SLOW && 32u * (uint32_t)s0 >= n_valid)
            break;
        // The read phase runs in stages across the PER sub-steps (all loads,
        // then all recursion arithmetic, then all table lookups, ...) so that
        // the sub-steps' latencies overlap.
        bool on[PER];
        uint32_t x1[PER], xp[PER], xq[PER], y[PER], xn[PER], ti[PER], o1[PER], o2[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int j = s0 / WG + i;
            const uint32_t m = (uint32_t)(s0 + i * WG) + (WG > 1 ? warp : 0u);
            on[i] = j < J && m < (uint32_t)M;   // uniform across the warp
            if (on[i]) {
                const int off = 32 * (s0 + i * WG);   // static part of 32m
                x1[i] = Sw[off + 1];    // word i+1
                xp[i] = Q[off];         // word i+pos   (Q = S + pos + 32*warp + lane)
                xq[i] = Q[off - 1];     // word i+pos-1
            }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i]) {
                const uint32_t yy = (r[s0 / WG + i] & P.mask) ^ x1[i];
                y[i] = yy ^ (yy << P.sh1) ^ (xp[i] >> P.sh2);
            }
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i])
                xn[i] = y[i] ^ tbl(Tb, 0u, y[i]);
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i])
                ti[i] = temper_index(xq[i]);
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (on[i]) {
                if (SLOW) {
                    o1[i] = temper_convert<0>(xn[i], ti[i], Tb);
                    o2[i] = temper_convert<1>(xn[i], ti[i], Tb);
                } else {
                    o1[i] = temper_convert<FMT>(xn[i], ti[i], Tb);
                }
            }
        if (WG > 1)
            __syncthreads();
        else
            __syncwarp();
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int j = s0 / WG + i;
            const uint32_t m = (uint32_t)(s0 + i * WG) + (WG > 1 ? warp : 0u);
            if (j < J && m < (uint32_t)M) {
                const int off = 32 * (s0 + i * WG);
                const uint32_t col = 32u * m + lane;
                const bool act = SLOW ? (col < n_valid) : (m + 1u < (uint32_t)M || lane <= last_lane);
                if (act) {
                    r[j] = xn[i];
                    Sw[off] = xn[i];
                    if (32u * m < P.mirror)
                        Sw[off + P.n] = xn[i];
                    if (SLOW)
                        slow_store(o1[i], o2[i], row_g + col, segs, s_first, s_end, out);
                    else
                        __stcs(ow + off, o1[i]);
                }
            }
        }
        if (WG > 1)
            __syncthreads();
        else
            __syncwarp();
    }
}

// ===========================================================================
// nfull consecutive full rows of one request, single warp, software-pipelined
// steps of W = 128 words (K = 4 sub-steps), with the tempering one row late.
//
// Late tempering.  The word i+pos that the recursion of number i picks up is
// the tempering word of number i+1, whose state word x_{i+1+N} is what the
// same lane reads as its neighbour word one row later.  So a lane looks up
// the tempering of number i+1 when it picks the word up, keeps it in T[m] for
// a row, and stores number i+1 when it reads x_{i+1+N}: one shared load less
// per number than reading word i+pos-1 again.  Row q of the run thus stores
// the numbers (q-1)N+1 .. qN; the last row's remaining numbers are stored
// after the loop.  Number 0 of the run is the one that column N-1 stores in
// the first row, from a T set up before it.
//
// Qp[m] is this lane's pick-up address for column group m, with the wrap at
// column N in it: a wrapped pick-up reads the new row's word at its own place
// in S, so nothing is mirrored behind the row.
//
// When N - pos >= 2W, the loads of step s+1 never touch a word that step s
// writes: word i+1 and the unwrapped pick-ups lie beyond step s's columns,
// and a wrapped pick-up of a column c < W(s+2) lands below c + pos - N < Ws.
// The same holds from the last step of a row to the first step of the next
// (its pick-ups end below pos + W <= N - W, where the last step begins at or
// above N - W).  So the loads of step s+1 are issued before the stores of
// step s, and one __syncwarp per step (after the stores) orders every store
// before the loads that read it two steps later.  The neighbour of column
// N-1 is column 0 of the new row (`x1_last` points there): written in step 0
// and read in step NS-2 >= 1 or later.  The loads issued during a row's last
// step are those of step 0 (the same addresses in every row); after the last
// row they are simply unused.  Before the first row these loads are made apart,
// and the numbers after the loop read neighbours' words too, which a run that
// follows at once (a request that ends with a row) overwrites in its step 0: a
// barrier before the loop orders both before step 0's stores.  Lanes past
// column N-1 in the last group compute on the words behind the row and write
// there; only their output store is predicated off.
//
// What bounds it (ncu, 1216 streams, 8 warps per SM, Mexp 11213): 6.03 LSU and
// 10.0 ALU instructions per 32 numbers, LSU data stage 91 % and ALU 70 % busy
// (the loop it replaced: 7.34 and 13.3).  Hence the late tempering and the
// wrapped addresses (LSU), the packed folds and the multiply for the left
// shift (ALU).  Only the packed tempering indices are kept for a row, a
// quarter register per column group: kept table words made the 44 groups of
// Mexp 44497 spill (0.98 against 0.86 ms).  The rows are unrolled because a
// row of three steps leaves its pointer and register moves exposed: one
// stream alone took 0.62 ms for 2^20 numbers with one row per pass, 0.52 with
// four.  All together: the uneven workload 4.72 -> 3.60 ms (1085 -> 1422
// Gnumbers/s, 0.84 of the HBM rate), 4096 x 2^18 at 12 warps per SM 1.02 ->
// 0.79 ms, one stream of 2^20 numbers 0.75 -> 0.52 ms; Mexp 44497, 1024 x
// 2^20, 1.15 -> 0.86 ms.
// ===========================================================================
__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Shared loads and stores at a compile-time offset from a 32-bit shared
// address: the offset is part of the instruction, so one address register
// serves a whole row.
template <int OFF>
__device__ __forceinline__ uint32_t lds_at(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(a), "n"(OFF) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts_at(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u32 [%0+%1], %2;" ::"r"(a), "n"(OFF), "r"(v) : "memory");
}

// f(0), f(1), .. f(N-1), the argument a compile-time constant.
template <class F, int... I>
__device__ __forceinline__ void static_for_impl(F&& f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F&& f)
{
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// Tempering indices of four words at once, as bytes 4 * index: the 16-bit and
// 8-bit folds run packed, two and four words to a register.  A byte permute
// then puts one of them under the table base tb, a multiple of 256, as the
// lookup's address (less the table's offset).  13 ALU instructions for four
// words in all, 16 one by one.
__device__ __forceinline__ uint32_t temper_pack(const uint32_t (&x)[4])
{
    const uint32_t u = __byte_perm(x[0], x[1], 0x5410) ^ __byte_perm(x[0], x[1], 0x7632);
    const uint32_t v = __byte_perm(x[2], x[3], 0x5410) ^ __byte_perm(x[2], x[3], 0x7632);
    return ((__byte_perm(u, v, 0x6420) ^ __byte_perm(u, v, 0x7531)) & 0x0F0F0F0Fu) * 4u;
}

template <int FMT>
__device__ __forceinline__ uint32_t finish(uint32_t v, uint32_t t)
{
    if (FMT == 0)
        return v ^ t;
    const uint32_t b = (v >> 9) ^ t;
    if (FMT == 1)
        return b;
    return __float_as_uint(__uint_as_float(b) - 1.0f);
}

template <int M, int FMT>
__device__ __forceinline__ void gen_rows_late(uint32_t* S, uint32_t* ow, const RowP& P, uint32_t lane,
                                              const uint32_t* __restrict__ Tb, uint32_t nfull)
{
    constexpr int K = 4;
    constexpr int NS = (M + K - 1) / K;   // steps per row (>= 3 here)
    constexpr int U = NS <= 3 ? 4 : 2;    // rows per pass of the unrolled loop
    constexpr int TT = FMT == 0 ? 64 : 128;   // byte offset of the tempering table
    const uint32_t N = P.n, last_lane = (N - 1u) & 31u;   // lane of column N-1 (group M-1)
    uint32_t sa = saddr(S + lane);
    uint32_t x1_last = lane >= last_lane ? saddr(S) : sa + 128u * (M - 1) + 4u;
    uint32_t tb = saddr(Tb);
    // the left shift as a multiply by a power of two that the compiler cannot
    // see through: the FMA pipe is idle, the ALU pipe is not
    uint32_t mul1 = 1u << P.sh1;
    asm volatile("" : "+r"(mul1), "+r"(sa), "+r"(x1_last), "+r"(tb));
    const uint32_t t0 = temper_index(S[P.pos - 1u]);
    uint32_t x1[K], xp[K];
    static_assert(M >= K, "step 0 fills all of x1 and xp");
    static_for<K>([&](auto ii) {
        constexpr int i = ii.value;
        const uint32_t p = 32u * i + lane + P.pos;
        x1[i] = lds_at<128 * i + 4>(sa);
        xp[i] = lds_at<0>(saddr(S + (p < N ? p : p - N)));
    });
    __syncwarp();   // these loads, and the last ones of a run before, come before step 0's stores
    uint32_t r[M], qa[M];
    uint32_t T[NS];   // the steps' tempering indices, packed
    static_for<M>([&](auto im) {
        constexpr int m = im.value;
        const uint32_t p = 32u * m + lane + P.pos;
        r[m] = lds_at<128 * m>(sa);
        qa[m] = saddr(S + (p < N ? p : p - N));
        asm volatile("" : "+r"(qa[m]));   // kept, not worked out again in the loop
    });
    static_for<NS>([&](auto is) { T[is.value] = 0u; });
    T[NS - 1] = (t0 & 15u) << (2 + 8 * ((M - 1) & 3));
    uint32_t* op = ow + 1 - (int)N;   // where column `lane` of this row stores
#pragma unroll U
    for (uint32_t q = 0; q < nfull; ++q, op += N) {
        const bool body = q != 0u;
        const bool last = lane == last_lane || (body && lane < last_lane);
        static_for<NS>([&](auto is) {
            constexpr int st = is.value, s0 = st * K;
            constexpr int n0 = (st + 1 < NS) ? s0 + K : 0;   // next step (next row's first)
            uint32_t y1[K], yp[K], xn[K], o[K], tw[K];
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value, m = n0 + i;
                if constexpr (m < M) {
                    if constexpr (m + 1 < M)
                        y1[i] = lds_at<128 * m + 4>(sa);
                    else
                        y1[i] = lds_at<0>(x1_last);
                    yp[i] = lds_at<0>(qa[m]);
                }
            });
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value;
                if constexpr (s0 + i < M)
                    tw[i] = lds_at<TT>(__byte_perm(T[st], tb, 0x7650 + i));
            });
            T[st] = temper_pack(xp);
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value, m = s0 + i;
                if constexpr (m < M) {
                    const uint32_t yy = (r[m] & P.mask) ^ x1[i];
                    const uint32_t y = yy ^ (yy * mul1) ^ (xp[i] >> P.sh2);
                    xn[i] = y ^ tbl(Tb, 0u, y);
                    o[i] = finish<FMT>(x1[i], tw[i]);
                }
            });
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value, m = s0 + i;
                if constexpr (m < M) {
                    r[m] = xn[i];
                    sts_at<128 * m>(sa, xn[i]);
                    if (m + 1 < M ? body : last)
                        __stcs(op + 32 * m, o[i]);
                }
            });
            __syncwarp();
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value;
                if constexpr (n0 + i < M) {
                    x1[i] = y1[i];
                    xp[i] = yp[i];
                }
            });
        });
    }
    // the last row's numbers after its first
    static_for<M>([&](auto im) {
        constexpr int m = im.value;
        const uint32_t v = lds_at<128 * m + 4>(sa);
        const uint32_t tw = lds_at<TT>(__byte_perm(T[m / K], tb, 0x7650 + m % K));
        if (m + 1 < M || lane < last_lane)
            __stcs(op + 32 * m, finish<FMT>(v, tw));
    });
}

// nfull consecutive full rows of one request for short states (M < 9, no
// 128-word step fits): the same late tempering and wrapped addresses, one
// 32-column sub-step at a time, each with the next sub-step's words read
// before its own are written.  That is exact while N - pos >= 64: none of
// those words is written by the current sub-step, and a wrapped pick-up lands
// on a column of an earlier, already written sub-step.
// What bounds it: the chain of a sub-step (lookup, store, barrier) at few
// warps, the LSU and ALU at many; 101 of 128 lanes work at Mexp 3217.
// Measured there against steps of 64 words read, passed and written: uneven
// workload unsplit 9.9 -> 5.6 ms, split in pieces of 701 932 6.4 -> 4.7 ms,
// 2432 equal streams at 16 warps per SM 721 -> 1098 Gnumbers/s.
template <int M, int FMT>
__device__ __forceinline__ void gen_rows_short(uint32_t* S, uint32_t* ow, const RowP& P, uint32_t lane,
                                               const uint32_t* __restrict__ Tb, uint32_t nfull)
{
    static_assert(M >= 3 && M <= 8, "two packed index registers, and a neighbour of column N-1 in time");
    constexpr int TT = FMT == 0 ? 64 : 128;
    constexpr int NT = (M + 3) / 4;
    const uint32_t N = P.n, last_lane = (N - 1u) & 31u;
    uint32_t sa = saddr(S + lane);
    uint32_t x1_last = lane >= last_lane ? saddr(S) : sa + 128u * (M - 1) + 4u;
    uint32_t tb = saddr(Tb);
    uint32_t mul1 = 1u << P.sh1;   // on the FMA pipe, as in gen_rows_late
    asm volatile("" : "+r"(mul1), "+r"(sa), "+r"(x1_last), "+r"(tb));
    // what other lanes write is read before the barrier (as in gen_rows_late);
    // the loop is 1.5 % faster for these loads standing first
    const uint32_t p0 = lane + P.pos, t0 = temper_index(S[P.pos - 1u]);
    uint32_t x1 = lds_at<4>(sa), xp = lds_at<0>(saddr(S + (p0 < N ? p0 : p0 - N)));
    __syncwarp();
    uint32_t r[M], qa[M], T[NT], xs[4 * NT];
    static_for<M>([&](auto im) {
        constexpr int m = im.value;
        const uint32_t p = 32u * m + lane + P.pos;
        r[m] = lds_at<128 * m>(sa);
        qa[m] = saddr(S + (p < N ? p : p - N));
        asm volatile("" : "+r"(qa[m]));
    });
    static_for<NT>([&](auto i) { T[i.value] = 0u; });
    static_for<4 * NT>([&](auto i) { xs[i.value] = 0u; });
    T[NT - 1] = (t0 & 15u) << (2 + 8 * ((M - 1) & 3));
    uint32_t* op = ow + 1 - (int)N;
#pragma unroll 4
    for (uint32_t q = 0; q < nfull; ++q, op += N) {
        const bool body = q != 0u;
        const bool last = lane == last_lane || (body && lane < last_lane);
        static_for<M>([&](auto im) {
            constexpr int m = im.value, n = m + 1 < M ? m + 1 : 0;
            uint32_t y1;
            if constexpr (n + 1 < M)
                y1 = lds_at<128 * n + 4>(sa);
            else
                y1 = lds_at<0>(x1_last);
            const uint32_t yp = lds_at<0>(qa[n]);
            const uint32_t yy = (r[m] & P.mask) ^ x1;
            const uint32_t y = yy ^ (yy * mul1) ^ (xp >> P.sh2);
            r[m] = y ^ tbl(Tb, 0u, y);
            const uint32_t tw = lds_at<TT>(__byte_perm(T[m / 4], tb, 0x7650 + m % 4));
            const uint32_t o = finish<FMT>(x1, tw);
            xs[m] = xp;
            sts_at<128 * m>(sa, r[m]);
            if (m + 1 < M ? body : last)
                __stcs(op + 32 * m, o);
            __syncwarp();
            x1 = y1;
            xp = yp;
        });
        static_for<NT>([&](auto i) {
            constexpr int b = 4 * i.value;
            const uint32_t x4[4] = {xs[b], xs[b + 1], xs[b + 2], xs[b + 3]};
            T[i.value] = temper_pack(x4);
        });
    }
    static_for<M>([&](auto im) {
        constexpr int m = im.value;
        const uint32_t v = lds_at<128 * m + 4>(sa);
        const uint32_t tw = lds_at<TT>(__byte_perm(T[m / 4], tb, 0x7650 + m % 4));
        if (m + 1 < M || lane < last_lane)
            __stcs(op + 32 * m, finish<FMT>(v, tw));
    });
}

template <int M, int FMT>
__device__ __forceinline__ void gen_full_rows(uint32_t* S, uint32_t* ow, const RowP& P, uint32_t lane,
                                              const uint32_t* __restrict__ Tb, uint32_t nfull)
{
    if constexpr (M < 9)
        gen_rows_short<M, FMT>(S, ow, P, lane, Tb, nfull);
    else
        gen_rows_late<M, FMT>(S, ow, P, lane, Tb, nfull);
}

// A row on the same layout (no mirror) with its numbers stored at once:
// columns 0 .. n_valid-1, in steps of 128 words, 64 for short states.  SLOW:
// the row crosses into another request and every lane finds its own;
// otherwise the row's numbers go to `ow`.
template <int M, int FMT, bool SLOW>
__device__ __forceinline__ void gen_row_part(uint32_t* S, uint32_t* ow, const RowP& P, uint32_t lane,
                                             const uint32_t* __restrict__ Tb, uint32_t n_valid,
                                             uint64_t row_g, const Segment* __restrict__ segs,
                                             uint32_t s_first, uint32_t s_end, uint32_t* __restrict__ out)
{
    constexpr int K = M < 9 ? 2 : 4;
    const uint32_t N = P.n;
    uint32_t* const Sw = S + lane;
#pragma unroll 1
    for (uint32_t c0 = 0; c0 < n_valid; c0 += 32u * K) {
        uint32_t xn[K], ti[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t c = c0 + 32u * i + lane;
            if (c0 + 32u * i < n_valid) {
                // lanes past column N-1 read in bounds and are not stored
                const uint32_t p = c + P.pos, pw = p < N ? p : p - N;
                const uint32_t yy = (Sw[c0 + 32 * i] & P.mask) ^ S[c + 1u == N ? 0u : c + 1u];
                const uint32_t y = yy ^ (yy << P.sh1) ^ (S[pw] >> P.sh2);
                xn[i] = y ^ tbl(Tb, 0u, y);
                ti[i] = temper_index(S[pw ? pw - 1u : N - 1u]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const uint32_t c = c0 + 32u * i + lane;
            if (c < n_valid) {
                S[c] = xn[i];
                if (SLOW)
                    slow_store(temper_convert<0>(xn[i], ti[i], Tb), temper_convert<1>(xn[i], ti[i], Tb),
                               row_g + c, segs, s_first, s_end, out);
                else
                    __stcs(ow + c0 + 32 * i, temper_convert<FMT>(xn[i], ti[i], Tb));
            }
        }
        __syncwarp();
    }
}

// Advances one stream whose N - pos >= 256 (>= 64 for short states) by the
// segments [s_begin, s_end), this warp alone.
template <int M>
__device__ __forceinline__ void run_item_late(const KParams& KP, const RowP& P, uint32_t* __restrict__ g,
                                              uint32_t* __restrict__ S, const Segment* __restrict__ segs,
                                              uint32_t s_begin, uint32_t s_end, uint32_t* __restrict__ out,
                                              uint32_t lane, const uint32_t* __restrict__ Tb)
{
    const uint32_t N = P.n;
    for (uint32_t c = lane; c < (KP.np >> 2); c += 32u)
        cp_async16(S + 4u * c, g + 4u * c);
    const Segment last = segs[s_end - 1u];
    uint32_t s = s_begin;
    Segment sg = segs[s];
    cp_async_wait_all();
    __syncwarp();
    const uint64_t total = last.g_start + last.count;
    uint64_t seg_end = sg.g_start + sg.count;
    uint64_t row = 0;
    while (row < total) {
        while (row >= seg_end) {
            sg = segs[++s];
            seg_end = sg.g_start + sg.count;
        }
        uint32_t* ow = out + sg.out_off + (row - sg.g_start) + lane;
        if (row + N <= seg_end) {
            // the rows that lie wholly inside this request, back to back
            const uint32_t nfull = (uint32_t)min((seg_end - row) / N, (uint64_t)0xFFFFFFFFu);
            if (sg.fmt == 0)
                gen_full_rows<M, 0>(S, ow, P, lane, Tb, nfull);
            else if (sg.fmt == 1)
                gen_full_rows<M, 1>(S, ow, P, lane, Tb, nfull);
            else
                gen_full_rows<M, 2>(S, ow, P, lane, Tb, nfull);
            row += (uint64_t)nfull * N;
        } else {
            const uint64_t left = total - row;
            const uint32_t n_valid = left < (uint64_t)N ? (uint32_t)left : N;
            if (total > seg_end)   // crosses into the next request
                gen_row_part<M, 0, true>(S, ow, P, lane, Tb, n_valid, row, segs, s, s_end, out);
            else if (sg.fmt == 0)
                gen_row_part<M, 0, false>(S, ow, P, lane, Tb, n_valid, row, segs, s, s_end, out);
            else if (sg.fmt == 1)
                gen_row_part<M, 1, false>(S, ow, P, lane, Tb, n_valid, row, segs, s, s_end, out);
            else
                gen_row_part<M, 2, false>(S, ow, P, lane, Tb, n_valid, row, segs, s, s_end, out);
            row += N;
        }
    }
    // stage out: oldest word first (see run_item)
    const uint32_t phase = (uint32_t)(total % N);
    for (uint32_t j = lane; j < N; j += 32u) {
        uint32_t c = phase + j;
        c = c >= N ? c - N : c;
        g[j] = S[c];
    }
    __syncwarp();
}

// Advances one stream by the segments [s_begin, s_end) of the work table.
// WG warps take part (WG = 1: this warp alone; WG = G: the whole CTA).
template <int M, int K, int WG>
__device__ __forceinline__ void run_item(const KParams& KP, const RowP& P, uint32_t* __restrict__ g,
                                         uint32_t* __restrict__ S, const Segment* __restrict__ segs,
                                         uint32_t s_begin, uint32_t s_end, uint32_t* __restrict__ out,
                                         uint32_t warp, uint32_t lane, const uint32_t* __restrict__ Tb)
{
    constexpr int J = (M + WG - 1) / WG;
    const uint32_t N = P.n;
    const uint32_t tid = WG > 1 ? threadIdx.x : lane;
    const uint32_t wk = WG > 1 ? warp : 0u;
    const uint32_t last_lane = (N - 1u) & 31u;   // lane of column N-1 (group M-1)

    // stage in: the state row (HBM) -> S through 16-byte cp.async
    for (uint32_t c = tid; c < (KP.np >> 2); c += 32u * WG)
        cp_async16(S + 4u * c, g + 4u * c);
    cp_async_wait_all();
    if (WG > 1)
        __syncthreads();
    else
        __syncwarp();
    uint32_t r[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const uint32_t c = 32u * (wk + (uint32_t)(j * WG)) + lane;
        r[j] = c < N ? S[c] : 0u;
    }
    // mirror: columns 0 .. P.mirror-1 again at S[N ..]
    for (uint32_t c = tid; c < P.mirror; c += 32u * WG) {
        const uint32_t v = S[c];
        S[N + c] = v;
    }
    if (WG > 1)
        __syncthreads();
    else
        __syncwarp();

    uint32_t* Sw = S + 32u * wk + lane;
    const uint32_t* Q = S + P.pos + 32u * wk + lane;
    const Segment last = segs[s_end - 1u];
    const uint64_t total = last.g_start + last.count;
    // The current request stays in registers: rows only touch the table
    // when they cross into the next request (a dependent global load per row
    // would put an L2 round trip on every row's critical path).
    uint32_t s = s_begin;
    Segment sg = segs[s];
    uint64_t seg_end = sg.g_start + sg.count;
    uint64_t row = 0;
    while (row < total) {
        while (row >= seg_end) {
            sg = segs[++s];
            seg_end = sg.g_start + sg.count;
        }
        if (row + N <= seg_end) {
            // The rows that lie wholly inside this request run back to back:
            // per row only the output pointer moves.
            const uint32_t nfull = (uint32_t)min((seg_end - row) / N, (uint64_t)0xFFFFFFFFu);
            uint32_t* ow = out + sg.out_off + (row - sg.g_start) + 32u * wk + lane;
            if (sg.fmt == 0) {
                for (uint32_t q = 0; q < nfull; ++q, ow += N)
                    gen_row<M, K, WG, 0, false>(r, S, Sw, ow, Q, P, wk, lane, Tb, last_lane, N, row,
                                                segs, s, s_end, out);
            } else if (sg.fmt == 1) {
                for (uint32_t q = 0; q < nfull; ++q, ow += N)
                    gen_row<M, K, WG, 1, false>(r, S, Sw, ow, Q, P, wk, lane, Tb, last_lane, N, row,
                                                segs, s, s_end, out);
            } else {
                for (uint32_t q = 0; q < nfull; ++q, ow += N)
                    gen_row<M, K, WG, 2, false>(r, S, Sw, ow, Q, P, wk, lane, Tb, last_lane, N, row,
                                                segs, s, s_end, out);
            }
            row += (uint64_t)nfull * N;
        } else {
            // a row that crosses into the next request, or the partial last row
            const uint64_t left = total - row;
            const uint32_t n_valid = left < (uint64_t)N ? (uint32_t)left : N;
            gen_row<M, K, WG, 0, true>(r, S, Sw, nullptr, Q, P, wk, lane, Tb, last_lane, n_valid,
                                       row, segs, s, s_end, out);
            row += N;
        }
    }

    // stage out: oldest word first, x_total .. x_{total+N-1}; the column of
    // x_{total+j} is (total + j) mod N
    const uint32_t phase = (uint32_t)(total % N);
    for (uint32_t j = tid; j < N; j += 32u * WG) {
        uint32_t c = phase + j;
        c = c >= N ? c - N : c;
        g[j] = S[c];
    }
    if (WG > 1)
        __syncthreads();
    else
        __syncwarp();
}

// One stream on one warp: the late-tempering loops where their steps fit
// (N - pos >= 256, short states always), else the general one.
template <int M, int K>
__device__ __forceinline__ void run_single(const KParams& KP, const RowP& P, uint32_t* __restrict__ g,
                                           uint32_t* __restrict__ S, const Segment* __restrict__ segs,
                                           uint32_t s_begin, uint32_t s_end, uint32_t* __restrict__ out,
                                           uint32_t warp, uint32_t lane, const uint32_t* __restrict__ Tb)
{
    if constexpr (M < 9) {   // 32 K <= N - pos, so N - pos >= 64
        run_item_late<M>(KP, P, g, S, segs, s_begin, s_end, out, lane, Tb);
    } else {
        if (P.n - P.pos >= 256u)
            run_item_late<M>(KP, P, g, S, segs, s_begin, s_end, out, lane, Tb);
        else
            run_item<M, K, 1>(KP, P, g, S, segs, s_begin, s_end, out, warp, lane, Tb);
    }
}

// Claims.  The n items (longest first) are dealt to n_groups lists, one per
// SM, in snake order: list g's k-th item is k n_groups + g for even k and
// k n_groups + (n_groups - 1 - g) for odd k.  A warp takes its own SM's next
// item, and when that list is used up helps with a list that still has more
// items than its SM has warps (those few its own warps take in one round), or
// with a list whose SM runs no CTA of this launch.  One list for the whole
// device let the SMs whose warps happened to be first take more of the last
// items than others: 1024 equal streams put 8 warps on some SMs and 5 on
// others, and 4096 at 16 warps per SM ended anywhere between 0.83 and 0.95 ms.
// Launches of short streams have one list all the same (one_claim_list).
constexpr uint32_t kNoItem = 0xFFFFFFFFu;
constexpr uint32_t kPresent = 0x80000000u;   // a list's counter: its SM runs a CTA of the launch

struct Claims {
    uint32_t* counters;   // n_groups counters, each with its kPresent bit
    uint32_t n;           // items
    uint32_t n_groups;
    uint32_t spare;       // warps per SM: what a present SM is left to do itself
    uint32_t group;       // the list this warp takes from
};

__device__ __forceinline__ uint32_t list_item(uint32_t k, uint32_t g, uint32_t n_groups)
{
    return k * n_groups + ((k & 1u) ? n_groups - 1u - g : g);
}

// This warp's view of the lists; one warp of each CTA marks its list.
__device__ __forceinline__ Claims claims_begin(uint32_t* counters, uint32_t n, uint32_t n_groups)
{
    Claims c;
    c.counters = counters;
    c.n = n;
    c.n_groups = n_groups;
    c.spare = (gridDim.x * (blockDim.x >> 5) + n_groups - 1u) / n_groups;
    // fewer CTAs than SMs: one list per CTA
    c.group = gridDim.x <= n_groups ? blockIdx.x : sm_id() % n_groups;
    if (threadIdx.x == 0u)
        atomicOr(counters + c.group, kPresent);
    return c;
}

// The warp's next item, or kNoItem when there is none it should take.  Every
// round either returns or finds its list used up for good (counters only
// grow) and moves on, so the rounds are bounded by the number of lists.
__device__ __forceinline__ uint32_t claim_item(Claims& c, uint32_t lane)
{
    for (;;) {
        uint32_t k = 0;
        if (lane == 0u)
            k = atomicAdd(c.counters + c.group, 1u) & ~kPresent;
        k = __shfl_sync(MTGP_FULL, k, 0);
        const uint32_t it = list_item(k, c.group, c.n_groups);
        if (it < c.n)
            return it;
        uint32_t next = kNoItem;
        for (uint32_t b = 1u; b < c.n_groups && next == kNoItem; b += 32u) {
            uint32_t j = c.group + b + lane;
            j = j >= c.n_groups ? j - c.n_groups : j;
            bool has = false;
            if (b + lane < c.n_groups) {
                const uint32_t v = *(volatile uint32_t*)(c.counters + j);
                const uint32_t ahead = (v & kPresent) ? c.spare : 0u;
                has = list_item((v & ~kPresent) + ahead, j, c.n_groups) < c.n;
            }
            const uint32_t B = __ballot_sync(MTGP_FULL, has);
            if (B)
                next = __shfl_sync(MTGP_FULL, j, __ffs(B) - 1);
        }
        if (next == kNoItem)
            return kNoItem;
        c.group = next;
    }
}

// Resident CTAs the compiler leaves registers for in mtgp_fast_kernel: 12 warps per SM for the
// smaller states (168 registers), 8 for the larger ones, which keep three
// words per column group.  At 16 warps (128 registers) the late loop spilled
// and ran at 1190 instead of 1400 Gnumbers/s (2432 equal streams, Mexp 11213).
// Short states, with a chain of 32-column sub-steps to hide, run best at 16
// (2432 equal streams at Mexp 3217: 1098 Gnumbers/s; at 24 and 32 warps per SM
// the loop spills and runs at 840).
constexpr int fast_min_ctas(int M, int G)
{
    return (M < 9 ? 16 : M < 16 ? 12 : 8) / G;
}

// Persistent kernel.  Phase 1: the CTA claims the longest streams (items
// [0, n_coop) of the table, sorted longest first) one at a time and its G
// warps advance each together.  Phase 2: every warp claims the remaining
// items [n_coop, n_items) one by one and advances each alone.
#define MTGP_KERNEL_PARAMS                                                                       \
    uint32_t *__restrict__ states, uint32_t n_streams, const WorkItem *__restrict__ items,       \
        const Segment *__restrict__ segs, uint32_t n_items, uint32_t n_coop,                     \
        uint32_t *__restrict__ counters, uint32_t *__restrict__ out, int *__restrict__ err,      \
        uint64_t *__restrict__ trace, const KSet *__restrict__ sets,                             \
        const uint32_t *__restrict__ set_of, uint32_t n_groups
template <int M, int K, int G>
__global__ void __launch_bounds__(G * 32, fast_min_ctas(M, G)) mtgp_fast_kernel(const KParams P, MTGP_KERNEL_PARAMS)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ uint32_t s_claim;
    // Tables: Tb[0] holds the handle's set; with per-stream sets each warp
    // loads its stream's tables into its own Tb[warp] (256-byte rows: every
    // table is 64-byte aligned, entry k in bank k, and the address of a row ends
    // in a zero byte, under which the late loops put a packed tempering index).
    __shared__ __align__(256) uint32_t Tb[G][64];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    if (threadIdx.x < 16) {
        Tb[0][threadIdx.x] = P.rec[threadIdx.x];
        Tb[0][16 + threadIdx.x] = P.tmp[threadIdx.x];
        Tb[0][32 + threadIdx.x] = P.flt[threadIdx.x];
    }
    __syncthreads();
    const RowP R0 = {P.n, P.mask, P.pos, P.sh1, P.sh2, P.mirror};

    // The CTA-wide phase splits each parallel step's K sub-steps over the G
    // warps, so it exists only for K >= G and for handles with one parameter
    // set; otherwise every item is a single-warp item.
    const uint32_t first_single = (K >= G && !sets) ? n_coop : 0u;
    if constexpr (K >= G) {
    while (n_coop != 0u && !sets) {
        if (threadIdx.x == 0)
            s_claim = atomicAdd(&counters[0], 1u);
        __syncthreads();
        const uint32_t it = s_claim;
        __syncthreads();
        if (it >= n_coop)
            break;
        const WorkItem w = items[it];
        if (w.stream >= n_streams || w.nseg == 0) {
            if (threadIdx.x == 0)
                atomicOr(err, 1);
            continue;
        }
        const uint64_t t0 = trace ? global_ns() : 0;
        run_item<M, K, G>(P, R0, states + (size_t)w.stream * P.np, smem, segs, w.seg_begin,
                          w.seg_begin + w.nseg, out, warp, lane, Tb[0]);
        if (trace && threadIdx.x == 0)
            trace_item(trace, it, t0, segs, w);
    }
    }

    uint32_t* S = smem + warp * fast_smem_words(P.n, P.mirror);
    // No more items than warps: each warp has its item by its place, one warp
    // of every CTA before a second one of any, and no counter is touched.
    const bool placed = first_single == 0u && items_placed(n_items, gridDim.x, G);
    Claims claims;
    if (!placed)
        claims = claims_begin(counters + 1, n_items - first_single, n_groups);
    for (bool more = true; more;) {
        uint32_t it;
        if (placed) {
            it = warp * gridDim.x + blockIdx.x;
            more = false;
            if (it >= n_items)
                break;
        } else {
            it = claim_item(claims, lane);
            if (it == kNoItem)
                break;
            it += first_single;
        }
        const WorkItem w = items[it];
        if (w.stream >= n_streams || w.nseg == 0) {
            if (lane == 0)
                atomicOr(err, 1);
            continue;
        }
        const uint64_t t0 = trace ? global_ns() : 0;
        if (sets) {
            // this stream's own parameter set
            const KSet& ks = sets[set_of[w.stream]];
            const RowP R = {P.n, P.mask, ks.pos, ks.sh1, ks.sh2, ks.mirror};
            if (lane < 16u) {
                Tb[warp][lane] = ks.rec[lane];
                Tb[warp][16u + lane] = ks.tmp[lane];
                Tb[warp][32u + lane] = ks.flt[lane];
            }
            __syncwarp();
            run_single<M, K>(P, R, states + (size_t)w.stream * P.np, S, segs, w.seg_begin,
                             w.seg_begin + w.nseg, out, warp, lane, Tb[warp]);
        } else {
            run_single<M, K>(P, R0, states + (size_t)w.stream * P.np, S, segs, w.seg_begin,
                             w.seg_begin + w.nseg, out, warp, lane, Tb[0]);
        }
        if (trace && lane == 0)
            trace_item(trace, it, t0, segs, w);
    }
}

// Without the late-tempering loops: for steps of 256 words (K = 8) and where
// general_rows chooses it.  Its loops need few registers, so the compiler is
// left to choose (64 to 128, 16 to 32 warps per SM).  In one kernel with claims
// by place or from lists per SM the K = 8 loops came out 5 to 18 % slower (8
// warps per SM, 4096 x 2^16 at Mexp 11213: 334 us, 377 there), so items are
// claimed from one list, counters[1], always.
template <int M, int K, int G>
__global__ void __launch_bounds__(G * 32) mtgp_general_kernel(const KParams P, MTGP_KERNEL_PARAMS)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ uint32_t s_claim;
    __shared__ __align__(64) uint32_t Tb[G][48];   // 192-byte rows: every table starts on a 64-byte boundary
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    if (threadIdx.x < 16) {
        Tb[0][threadIdx.x] = P.rec[threadIdx.x];
        Tb[0][16 + threadIdx.x] = P.tmp[threadIdx.x];
        Tb[0][32 + threadIdx.x] = P.flt[threadIdx.x];
    }
    __syncthreads();
    const RowP R0 = {P.n, P.mask, P.pos, P.sh1, P.sh2, P.mirror};
    const uint32_t first_single = (K >= G && !sets) ? n_coop : 0u;
    if constexpr (K >= G) {
    for (; !sets;) {
        if (threadIdx.x == 0)
            s_claim = atomicAdd(&counters[0], 1u);
        __syncthreads();
        const uint32_t it = s_claim;
        __syncthreads();
        if (it >= n_coop)
            break;
        const WorkItem w = items[it];
        if (w.stream >= n_streams || w.nseg == 0) {
            if (threadIdx.x == 0)
                atomicOr(err, 1);
            continue;
        }
        const uint64_t t0 = trace ? global_ns() : 0;
        run_item<M, K, G>(P, R0, states + (size_t)w.stream * P.np, smem, segs, w.seg_begin,
                          w.seg_begin + w.nseg, out, warp, lane, Tb[0]);
        if (trace && threadIdx.x == 0)
            trace_item(trace, it, t0, segs, w);
    }
    }
    uint32_t* S = smem + warp * fast_smem_words(P.n, P.mirror);
    for (;;) {
        uint32_t it = 0;
        if (lane == 0)
            it = first_single + atomicAdd(&counters[1], 1u);
        it = __shfl_sync(MTGP_FULL, it, 0);
        if (it >= n_items)
            break;
        const WorkItem w = items[it];
        if (w.stream >= n_streams || w.nseg == 0) {
            if (lane == 0)
                atomicOr(err, 1);
            continue;
        }
        const uint64_t t0 = trace ? global_ns() : 0;
        if (sets) {
            // this stream's own parameter set
            const KSet& ks = sets[set_of[w.stream]];
            const RowP R = {P.n, P.mask, ks.pos, ks.sh1, ks.sh2, ks.mirror};
            if (lane < 16u) {
                Tb[warp][lane] = ks.rec[lane];
                Tb[warp][16u + lane] = ks.tmp[lane];
                Tb[warp][32u + lane] = ks.flt[lane];
            }
            __syncwarp();
            run_item<M, K, 1>(P, R, states + (size_t)w.stream * P.np, S, segs, w.seg_begin,
                              w.seg_begin + w.nseg, out, warp, lane, Tb[warp]);
        } else {
            run_item<M, K, 1>(P, R0, states + (size_t)w.stream * P.np, S, segs, w.seg_begin,
                              w.seg_begin + w.nseg, out, warp, lane, Tb[0]);
        }
        if (trace && lane == 0)
            trace_item(trace, it, t0, segs, w);
    }
}

}  // namespace mtgp
