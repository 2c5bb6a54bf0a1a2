// Generation kernel for launches of many short streams (brief_items).
//
// Streams of a few rows end before the unrolled row loops of mtgp_fast_kernel
// pay for their registers, which leave room for 8 to 16 warps per SM: what
// such a launch waits for is the chain of each item (claim, table entry, state
// in, a few steps, state out), and more warps hide it.  This kernel keeps
// nothing per column group, so one instantiation per step width serves every
// state size, and 80 registers give 24 warps per SM.
//
// What bounds it: that chain, and from about four rows an item the shared loads
// of the row loop (six per number; the late-tempering loops take three less).
// Measured as plans in the automatic shape, against mtgp_fast_kernel at its 8
// to 16 warps per SM (and in brackets its older rows at the tuned 16 to 32):
// 10 000 streams of 2^2 .. 2^8 numbers at Mexp 11213 21.2 -> 17.8 us (18.1), of
// 2^3 .. 2^10 at 44497 40.1 -> 25.9 (28.3), of 2^10 at 11213 36.0 -> 25.9 (29.4)
// and at 44497 65.5 -> 30.7 (59.4); 2538 of 2^8 at 11213 14.3 -> 8.1 (13.1).
// Reading a step ahead, as the other row loops do, took 126 registers: 10 000
// streams of 2^2 .. 2^9 at 23209 22.2 us at the 16 warps they leave room for.
#include "mtgp_fast.cuh"

namespace mtgp {

// Numbers of one request from column 0 of a row on, `count` <= 2^31 of them:
// whole rows, and then the part of a row that ends the stream.  Steps of 32 K
// columns (32 K <= N - pos), each read, passed and written.  Pick-ups past
// column N-1 have the wrap in their address: none or all of a step's lanes
// have it, except in one step per row.  S[N] repeats column 0 for the neighbour
// of column N-1; lanes past the last column read what lies behind the row.
template <int K, int FMT>
__device__ __forceinline__ void gen_rows_brief(uint32_t* S, uint32_t* ow, const RowP& P, uint32_t lane,
                                               const uint32_t* __restrict__ Tb, uint32_t count)
{
    const uint32_t N = P.n;
    const uint32_t sa = saddr(S + lane);
    for (;; count -= N, ow += N) {
        const uint32_t n = min(N, count);
#pragma unroll 1
        for (uint32_t c0 = 0; c0 < n; c0 += 32u * K) {
            uint32_t x0[K], x1[K], xp[K], xq[K], xn[K], o[K];
            const uint32_t a = sa + 4u * c0, p0 = c0 + P.pos;
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value;
                x0[i] = lds_at<128 * i>(a);
                x1[i] = lds_at<128 * i + 4>(a);
            });
            if (p0 + 32u * K <= N || p0 > N) {
                const uint32_t b = a + 4u * P.pos - (p0 > N ? 4u * N : 0u);
                static_for<K>([&](auto ii) {
                    constexpr int i = ii.value;
                    xp[i] = lds_at<128 * i>(b);
                    xq[i] = lds_at<128 * i - 4>(b);
                });
            } else {
                static_for<K>([&](auto ii) {
                    constexpr int i = ii.value;
                    const uint32_t p = p0 + 32u * i + lane, w = p < N ? p : p - N;
                    xp[i] = lds_at<0>(saddr(S + w));
                    xq[i] = lds_at<0>(saddr(S + (w ? w - 1u : N - 1u)));
                });
            }
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value;
                const uint32_t yy = (x0[i] & P.mask) ^ x1[i];
                const uint32_t y = yy ^ (yy << P.sh1) ^ (xp[i] >> P.sh2);
                xn[i] = y ^ tbl(Tb, 0u, y);
                o[i] = temper_convert<FMT>(xn[i], temper_index(xq[i]), Tb);
            });
            __syncwarp();
            static_for<K>([&](auto ii) {
                constexpr int i = ii.value;
                if (c0 + 32u * i + lane < n) {
                    sts_at<128 * i>(a, xn[i]);
                    __stcs(ow + c0 + 32 * i, o[i]);
                }
            });
            if (c0 == 0u && lane == 0u)
                sts_at<0>(a + 4u * N, xn[0]);
            __syncwarp();
        }
        if (count <= N)
            return;
    }
}

// Advances one stream by the segments [s_begin, s_end), this warp alone.
template <int K>
__device__ __forceinline__ void run_item_brief(const KParams& KP, const RowP& P, uint32_t* __restrict__ g,
                                               uint32_t* __restrict__ S, const Segment* __restrict__ segs,
                                               uint32_t s_begin, uint32_t s_end, uint32_t* __restrict__ out,
                                               uint32_t lane, const uint32_t* __restrict__ Tb)
{
    constexpr int kPart = K >= 4 ? 9 : 8;   // gen_row_part's steps: 128 words, or 64
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
        if (row + N <= seg_end || seg_end == total) {
            // up to the end of the stream, or the whole rows of this request
            uint32_t count = (uint32_t)min(seg_end - row, (uint64_t)0x80000000u);
            if (row + count != total)
                count -= count % N;
            uint32_t* ow = out + sg.out_off + (row - sg.g_start) + lane;
            if (sg.fmt == 0)
                gen_rows_brief<K, 0>(S, ow, P, lane, Tb, count);
            else if (sg.fmt == 1)
                gen_rows_brief<K, 1>(S, ow, P, lane, Tb, count);
            else
                gen_rows_brief<K, 2>(S, ow, P, lane, Tb, count);
            row += count;
        } else {
            // a row that crosses into the next request
            const uint64_t left = total - row;
            gen_row_part<kPart, 0, true>(S, nullptr, P, lane, Tb, left < (uint64_t)N ? (uint32_t)left : N, row, segs,
                                         s, s_end, out);
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

// Persistent kernel with the arguments of mtgp_fast_kernel.  Items go to warps
// by their place where there are no more of them than warps, else they are
// claimed from one list, counters[1].
template <int K, int G>
__global__ void __launch_bounds__(G * 32, 24 / G) mtgp_brief_kernel(const KParams P, uint32_t* __restrict__ states,
                                                           uint32_t n_streams,
                                                           const WorkItem* __restrict__ items,
                                                           const Segment* __restrict__ segs,
                                                           uint32_t n_items, uint32_t /* n_coop = 0 */,
                                                           uint32_t* __restrict__ counters,
                                                           uint32_t* __restrict__ out, int* __restrict__ err,
                                                           uint64_t* __restrict__ trace,
                                                           const KSet* __restrict__ sets,
                                                           const uint32_t* __restrict__ set_of,
                                                           uint32_t /* n_groups */)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ __align__(256) uint32_t Tb[G][64];   // as in mtgp_fast_kernel
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    if (threadIdx.x < 16) {
        Tb[0][threadIdx.x] = P.rec[threadIdx.x];
        Tb[0][16 + threadIdx.x] = P.tmp[threadIdx.x];
        Tb[0][32 + threadIdx.x] = P.flt[threadIdx.x];
    }
    __syncthreads();
    uint32_t* S = smem + warp * brief_smem_words(P.n);
    const uint32_t* T = sets ? Tb[warp] : Tb[0];
    RowP R = {P.n, P.mask, P.pos, P.sh1, P.sh2, P.mirror};
    const bool placed = items_placed(n_items, gridDim.x, G);
    for (bool more = true; more;) {
        uint32_t it = 0;
        if (placed) {
            it = warp * gridDim.x + blockIdx.x;
            more = false;
        } else {
            if (lane == 0u)
                it = atomicAdd(counters + 1, 1u);
            it = __shfl_sync(MTGP_FULL, it, 0);
        }
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
            R.pos = ks.pos;
            R.sh1 = ks.sh1;
            R.sh2 = ks.sh2;
            if (lane < 16u) {
                Tb[warp][lane] = ks.rec[lane];
                Tb[warp][16u + lane] = ks.tmp[lane];
                Tb[warp][32u + lane] = ks.flt[lane];
            }
            __syncwarp();
        }
        run_item_brief<K>(P, R, states + (size_t)w.stream * P.np, S, segs, w.seg_begin, w.seg_begin + w.nseg, out,
                          lane, T);
        if (trace && lane == 0)
            trace_item(trace, it, t0, segs, w);
    }
}

const void* brief_kernel_ptr(int K, int G)
{
    switch (K * 16 + G) {
    case 2 * 16 + 2: return (const void*)mtgp_brief_kernel<2, 2>;
    case 2 * 16 + 4: return (const void*)mtgp_brief_kernel<2, 4>;
    case 2 * 16 + 8: return (const void*)mtgp_brief_kernel<2, 8>;
    case 4 * 16 + 2: return (const void*)mtgp_brief_kernel<4, 2>;
    case 4 * 16 + 4: return (const void*)mtgp_brief_kernel<4, 4>;
    case 4 * 16 + 8: return (const void*)mtgp_brief_kernel<4, 8>;
    default: return nullptr;
    }
}

}  // namespace mtgp
