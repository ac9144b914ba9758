// k_query_set.cu -- the set stage (Algorithm 2's union per table and
// intersection across tables) of batches on the probe path, 32 * QW queries at
// a time.
//
// The probe kernels (k_probe.cuh, k_query_wide.cu) hand over every query whose
// R per-table cell masks all keep a hit cell, as those masks.  A block takes
// 32 * QW of them and transposes their masks in shared memory, so
// that T[r][cell] holds one bit per query: bit q = cell is hit in table r for
// query q.  A set i then needs one shared-memory read per table for all of
// them,
//     acc = registered(i) AND T[0][phi_0(i)] AND ... AND T[R-1][phi_{R-1}(i)],
// instead of one bit test per table and query.  A warp takes 256 consecutive
// IDs (32 lanes x 8), transposes each 32-ID x 32-query block of acc back with
// five shuffles, and every lane stores 8 words (one 32-byte sector) of its
// query's K-bit bitmap, which the gather expands.
//
// What bounds it: the shared-memory pipe.  32 IDs x 128 queries cost R 16-byte
// reads a lane at random cells (8.6 wavefronts each, measured) and 20 shuffles;
// on 2e4 document queries ncu shows 75% of the L1 and shared data pipe's
// wavefronts, 55% by shared memory alone, and 3 blocks an SM.  Measured, set
// stage with the probes before it, against one query per warp in the query
// kernel: 1e5 conjunctive queries over 1e5 documents (R = 8, B = 320) 11.7 ms
// -> 0.26 (probes) + 0.89; 1e4 over 5e5 documents (R = 6, B = 1000; no
// per-warp bitmap there, so a warp scans all IDs twice) 85.4 ms -> 0.03 +
// 0.54; 16 queries over 1e5 documents 202 us -> 28.
//
// Groups of 128 queries are the widest whose T leaves two blocks an SM room;
// with fewer than 65 or 33 queries narrower groups read less of T per ID.
#include <algorithm>

#include "rambo_impl.cuh"

namespace rgb {

constexpr int QS_THREADS = 256;
constexpr int QS_WARPS = QS_THREADS / 32;
constexpr uint32_t QS_IDS = 256;                  // IDs a warp takes at a time
constexpr size_t QS_SMEM_TWO = 100 * 1024;        // two blocks an SM
constexpr size_t QS_SMEM_MOST = 200 * 1024;
constexpr int QSW_THREADS = 1024;                 // wide layouts: one block an SM
constexpr int QSW_WARPS = QSW_THREADS / 32;

struct SetShared {
    uint32_t* dst[128];      // bitmaps of the group's queries
    uint32_t q[128];         // their indexes
    uint32_t cnt[128];       // their set bits in this item
    uint64_t warp[QSW_WARPS];
    bool last;
};

// 32x32 bit transpose across the warp: lane l's bit b becomes lane b's bit l.
// Step S swaps the S-bit halves of lane pairs S apart; a lane keeps the bits
// under its mask and takes the others from its partner's word, rotated.
struct Transpose {
    uint32_t keep[5];
    uint32_t rot[5];
    __device__ __forceinline__ explicit Transpose(unsigned lane) {
        const uint32_t low[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const unsigned S = 16u >> i;
            keep[i] = (lane & S) ? ~low[i] : low[i];
            rot[i] = (lane & S) ? 32 - S : S;
        }
    }
    template <int I>
    __device__ __forceinline__ uint32_t step(uint32_t x) const {
        const uint32_t y = __shfl_xor_sync(FULL, x, 16 >> I);
        return (x & keep[I]) | (__funnelshift_l(y, y, rot[I]) & ~keep[I]);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
        return step<4>(step<3>(step<2>(step<1>(step<0>(x)))));
    }
};

template <int QW>
__device__ __forceinline__ void load_t(const uint32_t* t, uint32_t (&v)[QW]) {
    if constexpr (QW == 1) {
        v[0] = *t;
    } else if constexpr (QW == 2) {
        const uint2 x = *reinterpret_cast<const uint2*>(t);
        v[0] = x.x, v[1] = x.y;
    } else {
        const uint4 x = *reinterpret_cast<const uint4*>(t);
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    }
}

// Queries [g * 32 * QW, ...) of the deferred list against IDs [256 * c0, 256 * c1).
template <int QW>
__device__ __forceinline__ void set_item(const IndexView& ix, const QueryOut& o, uint64_t nd, uint64_t g, uint32_t c0,
                                         uint32_t c1, uint32_t* T, SetShared& sh) {
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t W = ix.W, RS = ix.R * ix.S;
    const Transpose transpose(lane);
    const uint64_t slot0 = g * 32 * QW + lane;
    if (threadIdx.x < 32 * QW) {
        // where the queries' bitmaps go (null: no query)
        const uint64_t slot = g * 32 * QW + threadIdx.x;
        sh.dst[threadIdx.x] = slot < nd ? o.stage + slot * set_pitch(ix.K) : nullptr;
        sh.q[threadIdx.x] = slot < nd ? o.dq[slot] : 0u;
        sh.cnt[threadIdx.x] = 0;
    }
    // masks to T, up to four words of a table at a time (rows of S words, S = 1, 2 or a multiple of 4)
    const uint32_t vec = ix.S < 4 ? ix.S : 4, quads = ix.S / vec;
    for (uint32_t p = wid; p < ix.R * quads; p += QS_WARPS) {
        const uint32_t r = p / quads, w0 = (p - r * quads) * vec;
        uint32_t x[QW][4];
#pragma unroll
        for (int j = 0; j < QW; ++j) {
            const uint32_t* m = o.dmask + (slot0 + 32 * j) * RS + r * ix.S + w0;
            uint4 q = make_uint4(0, 0, 0, 0);
            if (slot0 + 32 * j < nd) {
                if (vec == 4) q = __ldg(reinterpret_cast<const uint4*>(m));
                else q.x = __ldg(m), q.y = vec == 2 ? __ldg(m + 1) : 0u;
            }
            x[j][0] = q.x, x[j][1] = q.y, x[j][2] = q.z, x[j][3] = q.w;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            if (w0 + v >= W || v >= (int)vec) break;
            uint32_t* t = T + ((r * W + w0 + v) * 32 + lane) * QW;
#pragma unroll
            for (int j = 0; j < QW; ++j) x[j][v] = transpose(x[j][v]);
            if constexpr (QW == 1) *t = x[0][v];
            else if constexpr (QW == 2) *reinterpret_cast<uint2*>(t) = make_uint2(x[0][v], x[1][v]);
            else *reinterpret_cast<uint4*>(t) = make_uint4(x[0][v], x[1][v], x[2][v], x[3][v]);
        }
    }
    __syncthreads();
    uint32_t tot[QW];
#pragma unroll
    for (int j = 0; j < QW; ++j) tot[j] = 0;
    const uint4* phi = reinterpret_cast<const uint4*>(ix.phi);
    for (uint32_t c = c0 + wid; c < c1; c += QS_WARPS) {
        uint32_t out[QW][8];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint64_t i0 = (uint64_t)c * QS_IDS + 128 * half + lane;
            uint4 ph[4];
            uint32_t reg[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint64_t i = i0 + 32 * u;
                const bool in = i < ix.K;
                ph[u] = in ? __ldg(phi + i) : make_uint4(0, 0, 0, 0);
                reg[u] = in ? __ldg(ix.reg + (i >> 5)) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t cell[8] = {ph[u].x & 0xffffu, ph[u].x >> 16, ph[u].y & 0xffffu, ph[u].y >> 16,
                                          ph[u].z & 0xffffu, ph[u].z >> 16, ph[u].w & 0xffffu, ph[u].w >> 16};
                uint32_t acc[QW];
#pragma unroll
                for (int j = 0; j < QW; ++j) acc[j] = (reg[u] >> lane) & 1u ? ~0u : 0u;
#pragma unroll
                for (int r = 0; r < RF; ++r) {
                    if (r < (int)ix.R) {
                        uint32_t v[QW];
                        load_t<QW>(T + (r * W * 32 + cell[r]) * QW, v);
#pragma unroll
                        for (int j = 0; j < QW; ++j) acc[j] &= v[j];
                    }
                }
#pragma unroll
                for (int j = 0; j < QW; ++j) out[j][4 * half + u] = transpose(acc[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < QW; ++j) {
            uint32_t* dst = sh.dst[32 * j + lane];
            if (!dst) continue;
            uint4* d = reinterpret_cast<uint4*>(dst + (uint64_t)c * 8);
            d[0] = make_uint4(out[j][0], out[j][1], out[j][2], out[j][3]);
            d[1] = make_uint4(out[j][4], out[j][5], out[j][6], out[j][7]);
#pragma unroll
            for (int u = 0; u < 8; ++u) tot[j] += __popc(out[j][u]);
        }
    }
#pragma unroll
    for (int j = 0; j < QW; ++j)
        if (tot[j]) atomicAdd(&sh.cnt[32 * j + lane], tot[j]);
    __syncthreads();
    if (threadIdx.x < 32 * QW && sh.cnt[threadIdx.x])
        atomicAdd(o.qcount + sh.q[threadIdx.x], sh.cnt[threadIdx.x]);
    __syncthreads();  // T and the counters are rewritten by the next item
}

template <int QW>
__device__ __forceinline__ void set_items(const IndexView& ix, const QueryOut& o, uint64_t nd, uint32_t* T,
                                          SetShared& sh) {
    // items = query groups x ID ranges.  A range is a whole number of the
    // block's steps (8 warps x 256 IDs); with few groups the ranges are
    // short, so that four items per block keep the grid even
    const uint32_t chunks = (uint32_t)((ix.K + QS_IDS - 1) / QS_IDS);
    const uint32_t steps = (chunks + QS_WARPS - 1) / QS_WARPS;
    const uint64_t groups = (nd + 32 * QW - 1) / (32 * QW);
    const uint64_t want = (4ull * gridDim.x + groups - 1) / groups;
    const uint32_t per = want < steps ? (steps + (uint32_t)want - 1) / (uint32_t)want : 1;
    const uint32_t ranges = (steps + per - 1) / per;
    for (uint64_t it = blockIdx.x; it < groups * ranges; it += gridDim.x) {
        const uint64_t g = it / ranges;
        const uint32_t r = (uint32_t)(it - g * ranges);
        const uint32_t c0 = min(chunks, r * per * QS_WARPS), c1 = min(chunks, (r + 1) * per * QS_WARPS);
        if (c0 < c1) set_item<QW>(ix, o, nd, g, c0, c1, T, sh);
    }
}

// Exclusive scan of n counts by one block (16 a thread and round), out[n] the
// total; the counts are read past L1 (other blocks added to them).
template <int THREADS>
__device__ __forceinline__ void scan_counts_block(const uint32_t* counts, uint64_t n, uint64_t* out, uint64_t carry,
                                                  unsigned long long* total_out, uint64_t* s_warp) {
    constexpr int PER = 16;
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (uint64_t base = 0; base < n; base += (uint64_t)THREADS * PER) {
        const uint64_t i0 = base + (uint64_t)threadIdx.x * PER;
        uint32_t v[PER];
        uint64_t sum = 0;
        if (i0 + PER <= n && (reinterpret_cast<uintptr_t>(counts) & 15) == 0) {
#pragma unroll
            for (int t = 0; t < PER; t += 4) {
                const uint4 x = __ldcg(reinterpret_cast<const uint4*>(counts + i0 + t));
                v[t] = x.x, v[t + 1] = x.y, v[t + 2] = x.z, v[t + 3] = x.w;
            }
        } else {
#pragma unroll
            for (int t = 0; t < PER; ++t) v[t] = i0 + t < n ? __ldcg(counts + i0 + t) : 0u;
        }
#pragma unroll
        for (int t = 0; t < PER; ++t) sum += v[t];
        uint64_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint64_t y = __shfl_up_sync(FULL, incl, off);
            if (lane >= (unsigned)off) incl += y;
        }
        if (lane == 31) s_warp[wid] = incl;
        __syncthreads();
        uint64_t pre = carry + incl - sum;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) {
            const uint64_t x = s_warp[w];
            if (w < (int)wid) pre += x;
            carry += x;
        }
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            if (i0 + t < n) out[i0 + t] = pre;
            pre += v[t];
        }
        __syncthreads();  // the warp totals are rewritten by the next round
    }
    if (threadIdx.x == 0) {
        out[n] = carry;
        if (total_out) *total_out = carry;
    }
}

// What every set kernel ends with: the words staged and queries served are
// noted, and (scan) the block that finishes last lays the answers out.
template <int THREADS>
__device__ __forceinline__ void set_finish(const IndexView& ix, const BatchView& b, const QueryOut& o, uint64_t nd,
                                           int scan, uint64_t* id_offsets, const uint64_t* base_dev,
                                           unsigned long long* total_out, DevStatus* st, SetShared& sh) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->cursor = nd * set_pitch(ix.K);  // words staged: by this launch, and (spare) by the whole batch
        st->spare[0] += nd * set_pitch(ix.K);
        st->stage_count[1] += nd;
    }
    if (!scan) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) sh.last = atomicAdd(&st->set_done, 1ull) == gridDim.x - 1;
    __syncthreads();
    if (!sh.last) return;
    __threadfence();
    scan_counts_block<THREADS>(o.qcount, b.n, id_offsets, base_dev ? *base_dev : 0, total_out, sh.warp);
}

__global__ void __launch_bounds__(QS_THREADS, 3)
    k_set(IndexView ix, BatchView b, QueryOut o, int qw, int scan, uint64_t* __restrict__ id_offsets,
          const uint64_t* __restrict__ base_dev, unsigned long long* __restrict__ total_out, DevStatus* st) {
    extern __shared__ __align__(16) uint32_t qs_smem[];
    __shared__ SetShared sh;
    bv_resolve(b);
    const uint64_t nd = st->n_handed;
    if (st->err != NO_ERR) return;
    if (nd) {
        // narrower groups when the batch does not fill a wide one
        if (qw >= 4 && nd > 64) set_items<4>(ix, o, nd, qs_smem, sh);
        else if (qw >= 2 && nd > 32) set_items<2>(ix, o, nd, qs_smem, sh);
        else set_items<1>(ix, o, nd, qs_smem, sh);
    }
    set_finish<QS_THREADS>(ix, b, o, nd, scan, id_offsets, base_dev, total_out, st, sh);
}

// Wide layouts (rows of thousands of cells, or more than eight tables): a bit
// per cell for each of 16 queries, in 16-bit words, of as many tables as fit
// shared memory; further tables take further passes over the IDs, which AND
// into the bitmaps of the pass before (every lane reads what it wrote).  A
// warp's transpose then serves two 32-ID units at once: their 16-bit words
// share a register.  Measured on 2e4 queries over 1e5 documents (B = 2e4, R = 4,
// one pass; 1.2e4 survive): 0.58 ms, and 0.28 for the probes before it, against
// 7.4 ms with each query's block testing every ID twice.  Groups of 32 queries
// would fit half the tables at a time and build T four times per ID range.
__device__ __forceinline__ void set_wide_item(const IndexView& ix, const QueryOut& o, uint64_t nd, uint64_t g,
                                              uint32_t c0, uint32_t c1, uint32_t per_pass, uint16_t* T, SetShared& sh) {
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t W = ix.W, RS = ix.R * ix.S, Bp = W * 32;
    const Transpose transpose(lane);
    const uint64_t slot0 = g * 16;
    if (threadIdx.x < 16) {
        const uint64_t slot = slot0 + threadIdx.x;
        sh.dst[threadIdx.x] = slot < nd ? o.stage + slot * set_pitch(ix.K) : nullptr;
        sh.q[threadIdx.x] = slot < nd ? o.dq[slot] : 0u;
        sh.cnt[threadIdx.x] = 0;
    }
    // this lane's query, and which 16 bits of a pair of mask words or units are its own
    const uint64_t my = slot0 + (lane & 15);
    const uint32_t half = lane >> 4;
    uint32_t tot = 0;
    // (a pass stays inside eight tables: their cells are one 16-byte read of the partition row)
    for (uint32_t r0 = 0; r0 < ix.R;) {
        const uint32_t r1 = min(min(ix.R, r0 + per_pass), (r0 / 8 + 1) * 8);
        const bool first = r0 == 0, last = r1 == ix.R;
        __syncthreads();  // the pass before has read T
        const uint32_t pairs = (W + 1) / 2;
        for (uint32_t p = wid; p < (r1 - r0) * pairs; p += QSW_WARPS) {
            const uint32_t r = p / pairs, w = (p - r * pairs) * 2;
            const uint32_t x =
                my < nd && w + half < W ? __ldg(o.dmask + my * RS + (r0 + r) * ix.S + w + half) : 0u;
            const uint32_t y = transpose(x);
            uint16_t* t = T + r * Bp + w * 32 + lane;
            t[0] = (uint16_t)y;
            if (w + 1 < W) t[32] = (uint16_t)(y >> 16);
        }
        __syncthreads();
        const uint4* phi = reinterpret_cast<const uint4*>(ix.phi) + r0 / 8;
        const uint32_t rows = ix.ps / 8, rr = r0 & 7, rn = r1 - r0;
        for (uint32_t c = c0 + wid; c < c1; c += QSW_WARPS) {
            uint32_t out[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                uint32_t acc[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint64_t i = (uint64_t)c * QS_IDS + 32 * (u + 4 * h) + lane;
                    const bool in = i < ix.K;
                    const uint4 ph = in ? __ldg(phi + i * rows) : make_uint4(0, 0, 0, 0);
                    const uint32_t reg = in && first ? __ldg(ix.reg + (i >> 5)) : ~0u;
                    const uint32_t cell[8] = {ph.x & 0xffffu, ph.x >> 16, ph.y & 0xffffu, ph.y >> 16,
                                              ph.z & 0xffffu, ph.z >> 16, ph.w & 0xffffu, ph.w >> 16};
                    uint32_t a = in && ((reg >> lane) & 1u) ? 0xffffu : 0u;
#pragma unroll
                    for (uint32_t r = 0; r < 8; ++r)
                        if (r >= rr && r < rr + rn) a &= T[(r - rr) * Bp + cell[r]];
                    acc[h] = a;
                }
                out[u] = transpose(acc[0] | (acc[1] << 16));
            }
            uint32_t* d = sh.dst[lane & 15];
            if (!d) continue;
            uint4* to = reinterpret_cast<uint4*>(d + (uint64_t)c * 8 + 4 * half);
            if (!first) {
                const uint4 was = *to;
                out[0] &= was.x, out[1] &= was.y, out[2] &= was.z, out[3] &= was.w;
            }
            *to = make_uint4(out[0], out[1], out[2], out[3]);
            if (last) tot += __popc(out[0]) + __popc(out[1]) + __popc(out[2]) + __popc(out[3]);
        }
        r0 = r1;
    }
    if (tot) atomicAdd(&sh.cnt[lane & 15], tot);
    __syncthreads();
    if (threadIdx.x < 16 && sh.cnt[threadIdx.x]) atomicAdd(o.qcount + sh.q[threadIdx.x], sh.cnt[threadIdx.x]);
    __syncthreads();  // the queries and counters are rewritten by the next item
}

__global__ void __launch_bounds__(QSW_THREADS, 1)
    k_set_wide(IndexView ix, BatchView b, QueryOut o, int per_pass, int scan, uint64_t* __restrict__ id_offsets,
               const uint64_t* __restrict__ base_dev, unsigned long long* __restrict__ total_out, DevStatus* st) {
    extern __shared__ __align__(16) uint32_t qs_smem[];
    __shared__ SetShared sh;
    bv_resolve(b);
    const uint64_t nd = st->n_handed;
    if (st->err != NO_ERR) return;
    if (nd) {
        // query groups x ID ranges of whole steps (32 warps x 256 IDs), two
        // items a block or more as long as there are steps to split
        const uint32_t chunks = (uint32_t)((ix.K + QS_IDS - 1) / QS_IDS);
        const uint32_t steps = (chunks + QSW_WARPS - 1) / QSW_WARPS;
        const uint64_t groups = (nd + 15) / 16;
        const uint64_t want = (2ull * gridDim.x + groups - 1) / groups;
        const uint32_t per = want < steps ? (steps + (uint32_t)want - 1) / (uint32_t)want : 1;
        const uint32_t ranges = (steps + per - 1) / per;
        for (uint64_t it = blockIdx.x; it < groups * ranges; it += gridDim.x) {
            const uint64_t g = it / ranges;
            const uint32_t r = (uint32_t)(it - g * ranges);
            const uint32_t c0 = min(chunks, r * per * QSW_WARPS), c1 = min(chunks, (r + 1) * per * QSW_WARPS);
            set_wide_item(ix, o, nd, g, c0, c1, (uint32_t)per_pass, reinterpret_cast<uint16_t*>(qs_smem), sh);
        }
    }
    set_finish<QSW_THREADS>(ix, b, o, nd, scan, id_offsets, base_dev, total_out, st, sh);
}

SetLaunch set_launch_shape(const IndexView& ix, int num_sms) {
    SetLaunch sl{};
    const bool wide = query_is_wide(ix.R, ix.S);
    const void* f = wide ? reinterpret_cast<const void*>(&k_set_wide) : reinterpret_cast<const void*>(&k_set);
    if (wide) {
        const size_t table = (size_t)ix.W * 32 * 2;  // 16 queries' bits of a table's cells
        sl.qw = (int)std::min<size_t>(ix.R, QS_SMEM_MOST / table);
        sl.smem = table * sl.qw;
    } else {
        const size_t one = (size_t)ix.R * ix.W * 32 * 4;  // a bit per cell for each of 32 queries
        sl.qw = 4 * one <= QS_SMEM_TWO ? 4 : 2 * one <= QS_SMEM_TWO ? 2 : one <= QS_SMEM_MOST ? 1 : 0;
        sl.smem = one * sl.qw;
    }
    if (!sl.qw) return sl;
    sl.wide = wide;
    int per_sm = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)QS_SMEM_MOST) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, wide ? QSW_THREADS : QS_THREADS, sl.smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        sl.qw = 0;
        return sl;
    }
    sl.blocks = per_sm * num_sms;
    return sl;
}

cudaError_t launch_set(const SetLaunch& sl, const IndexView& ix, const BatchView& b, const QueryOut& o, int scan,
                       uint64_t* id_offsets, const uint64_t* base_dev, unsigned long long* total_out, DevStatus* st,
                       cudaStream_t s) {
    if (b.n == 0 && !b.desc) return cudaSuccess;
    // no more blocks than there can be items (b.n is the capacity of a
    // descriptor batch): each one that has none still ends in a same-address
    // atomic, and 456 of them for 40 items cost 5 us
    const uint64_t step = (uint64_t)QS_IDS * (sl.wide ? QSW_WARPS : QS_WARPS);
    const uint64_t per = sl.wide ? 16 : 32 * (uint64_t)sl.qw;
    const uint64_t narrow = sl.wide ? 1 : b.n > 32 ? 2 : 1;  // groups of 32 up to 64 queries
    const uint64_t most = std::max((b.n + per - 1) / per, narrow) * ((ix.K + step - 1) / step);
    const unsigned blocks = (unsigned)((uint64_t)sl.blocks < most ? (uint64_t)sl.blocks : most);
    if (sl.wide)
        k_set_wide<<<blocks, QSW_THREADS, sl.smem, s>>>(ix, b, o, sl.qw, scan, id_offsets, base_dev, total_out, st);
    else
        k_set<<<blocks, QS_THREADS, sl.smem, s>>>(ix, b, o, sl.qw, scan, id_offsets, base_dev, total_out, st);
    return cudaGetLastError();
}

}  // namespace rgb
