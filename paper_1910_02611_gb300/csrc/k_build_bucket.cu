// k_build_bucket.cu -- construction (Algorithm 1, Sec. 3.1) with every key
// hashed once per input chunk.
//
// The windowed build (k_build.cu) keeps one L2-sized slice of the rows
// resident while the whole input streams past, so every key is extracted and
// hashed once per window.  Here a scatter pass hashes each key of a chunk of
// the input once, turns every (table, hash) bit it sets into a 4-byte update
// record -- the bit's offset inside its window of the rows -- and files the
// records into one bucket per window (a block-local counting sort in shared
// memory, then one reservation per window and block).  An apply pass then
// takes the windows one at a time and ORs their records into the rows with
// fire-and-forget atomics, so each window stays resident in L2 while it is
// written.  Setting bits is order-free, so the bits equal every other build's.
#include "rambo_impl.cuh"

namespace rgb {

constexpr int BK_THREADS = 512;
constexpr int BK_APPLY_THREADS = 256;
constexpr int BK_WARPS = BK_THREADS / 32;
constexpr uint32_t BK_SLOTS = 32;                             // most records a thread files per step
constexpr uint32_t BK_TILE_RECORDS = BK_THREADS * BK_SLOTS;   // most records of a block's step
constexpr uint32_t BK_MAX_WINDOWS = 4096;

// largest t in [lo, n) with off[t] <= pos (off[lo] is)
__device__ __forceinline__ uint64_t bk_find_item(const uint64_t* __restrict__ off, uint64_t lo, uint64_t n,
                                                 uint64_t pos) {
    uint64_t hi = n;
    while (hi - lo > 1) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (__ldg(off + mid) <= pos) lo = mid;
        else hi = mid;
    }
    return lo;
}

// How global rows fall into windows of rows_per_win rows.
struct WindowMap {
    uint64_t rows_per_win;
    // all rows below 2^32 and whole 2^unit rows a window: window of row g =
    // high word of magic * (g >> unit), magic = ceil(2^32 / (rows_per_win >>
    // unit)).  Exact while (g >> unit) * (rows_per_win >> unit) < 2^32 for
    // every g (Lemire, Kaser and Kurz, "Faster remainder by direct
    // computation", 2019); 0: divide
    uint32_t magic, unit;
};

// The update records of one key (hashed to y, its set's cells in `cell`):
// f(window, offset in the window) for every table and hash.  M32: row numbers
// fit 32 bits, windows come from the multiplication, and ETA is eta.
template <int RT, int ETA, bool M32, class F>
__device__ __forceinline__ void bk_records(const IndexView& ix, const HashParams& hp, const WindowMap& wm, uint64_t y,
                                           const uint4 (&cell)[RT / 8], F f) {
    const uint32_t bits = ix.S * 32, m = (uint32_t)ix.m, rows = (uint32_t)wm.rows_per_win;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        if (r < (int)ix.R) {
            const uint4 h = cell[r / 8];
            const uint32_t pair = (r & 6) == 0 ? h.x : (r & 6) == 2 ? h.y : (r & 6) == 4 ? h.z : h.w;
            const uint32_t c = (r & 1) ? pair >> 16 : pair & 0xffffu;  // word * 32 + bit of the row
#pragma unroll
            for (int j = 0; j < ETA; ++j) {
                if (M32 || j < (int)ix.eta) {  // (M32: ETA = eta)
                    // (at most 2^32 rows a table: the position is in the product's high word)
                    const uint32_t pos = (uint32_t)((hp.s[r][j] * y) >> 32) >> (ix.shift - 32);
                    if constexpr (M32) {
                        const uint32_t g = r * m + pos;  // global row
                        const uint32_t win = __umulhi(wm.magic, g >> wm.unit);
                        f(win, (g - win * rows) * bits + c);
                    } else {
                        const uint64_t g = (uint64_t)r * ix.m + pos;
                        const uint32_t win = (uint32_t)(g / wm.rows_per_win);
                        f(win, (uint32_t)(g - (uint64_t)win * wm.rows_per_win) * bits + c);
                    }
                }
            }
        }
    }
}

// Scatter: a block takes a contiguous run of key positions, KT a thread and
// step.  Each step it counts its records per window (shared-memory atomics),
// scans the counts into block-local offsets, reserves each window's share of
// its bucket with one global atomic, then walks the same keys again (their
// hashes are kept, the positions recomputed) and places every record at its
// window's offset in shared memory; the windows' runs leave as consecutive
// words, `run` lanes a window.  Filing the records needs no other staging, so
// a record costs two shared atomics, one store and one load.  A bucket that would overflow sets *overflow
// instead (the caller then files the chunk again).
//
// What bounds it: instruction issue (64% of the slots with 64 windows), then the
// shared-memory pipe (55%: the atomics and the scattered stores; 76% with 8
// windows, where a warp's lanes meet on the same counters).  Measured on 2e9 k-mers
// with R * eta = 12 (2.4e10 records, 128 windows): 181 -> 60.6 ms.  Staging
// every record with its window, two blocks of 256 threads an SM and a search
// for the item every step made up the 181; one multiplication for the window
// instead of a 64-bit one took 74 to 67, and loops over exactly eta hashes 67
// to 60.6.
template <int RT, int KT, int ETA, bool M32>
__global__ void __launch_bounds__(BK_THREADS, 2)
    k_bucket_scatter(IndexView ix, HashParams hp, BatchView b, uint64_t p_lo, uint64_t p_hi, WindowMap wm,
                     uint32_t n_win, uint32_t run, uint64_t cap, uint32_t* __restrict__ rec,
                     unsigned long long* __restrict__ fill, unsigned long long* overflow, const DevStatus* st) {
    extern __shared__ __align__(16) unsigned char bk_smem[];
    uint32_t* s_srt = reinterpret_cast<uint32_t*>(bk_smem);                                       // records by window
    unsigned long long* s_dst = reinterpret_cast<unsigned long long*>(s_srt + BK_TILE_RECORDS);  // [n_win] where its run goes
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_dst + n_win);                                 // [n_win] records, then next slot
    uint32_t* s_off = s_cnt + n_win;                                                               // [n_win] first slot
    __shared__ uint32_t s_wsum[BK_WARPS];
    if (st->err != NO_ERR) return;
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // each thread scans a contiguous run of the window counters
    const uint32_t wper = (n_win + BK_THREADS - 1) / BK_THREADS;
    const uint32_t wlo = min(n_win, threadIdx.x * wper), whi = min(n_win, wlo + wper);
    constexpr uint64_t span = (uint64_t)KT * BK_THREADS;
    // this block's positions, in whole steps
    const uint64_t steps = (p_hi - p_lo + span - 1) / span;
    const uint64_t first = p_lo + steps * blockIdx.x / gridDim.x * span;
    const uint64_t end = min(p_hi, p_lo + steps * (blockIdx.x + 1) / gridDim.x * span);
    // the item holding this thread's position: searched once, then walked forward
    uint64_t t = 0, t_end = 0;
    uint4 row[RT / 8];
    auto enter = [&](uint64_t item) {
        t = item;
        t_end = __ldg(b.offsets + t + 1) - b.off0;
    };
    auto cells = [&]() {
        const uint4* ph = reinterpret_cast<const uint4*>(ix.phi + __ldg(b.set_ids + t) * ix.ps);
#pragma unroll
        for (int h = 0; h < RT / 8; ++h) row[h] = __ldg(ph + h);
    };
    if (first < end) {
        const uint64_t p = min(first + (uint64_t)threadIdx.x * KT, end - 1);
        enter(bk_find_item(b.offsets, 0, b.n, p + b.off0));
        cells();
    }
    for (uint64_t p0 = first; p0 < end; p0 += span) {
        for (uint32_t w = threadIdx.x; w < n_win; w += BK_THREADS) s_cnt[w] = 0;
        __syncthreads();
        // this thread's keys: hashes and cells, and their records counted
        uint64_t y[KT];
        uint4 cell[KT][RT / 8];
        uint32_t have = 0;
#pragma unroll
        for (int u = 0; u < KT; ++u) {
            const uint64_t p = p0 + (uint64_t)threadIdx.x * KT + u;
            if (p >= end) continue;
            if (p >= t_end) {
                // the item holding p: mostly the next one, else a search (short items)
                enter(t + 1);
                if (p >= t_end) enter(bk_find_item(b.offsets, t, b.n, p + b.off0));
                cells();
            }
            if (b.seq && p + b.k > t_end) continue;  // window runs past the end of this set's sequence
            if (b.skipn && !window_resolved(b.nmask, p, b.k)) continue;
            uint64_t key;
            if (b.seq) {
                key = kmer_at(b.packed, p, b.k);
                if (b.canon) key = canonical_kmer(key, b.k);
            } else {
                key = __ldg(b.keys + p);
            }
            y[u] = mix64(key);
#pragma unroll
            for (int h = 0; h < RT / 8; ++h) cell[u][h] = row[h];
            have |= 1u << u;
            bk_records<RT, ETA, M32>(ix, hp, wm, y[u], cell[u], [&](uint32_t win, uint32_t) { atomicAdd(&s_cnt[win], 1u); });
        }
        __syncthreads();
        // block-local offsets of the windows, and each window's share of its
        // bucket reserved with one atomic
        uint32_t sum = 0;
        for (uint32_t w = wlo; w < whi; ++w) sum += s_cnt[w];
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t v = __shfl_up_sync(FULL, incl, off);
            if (lane >= (unsigned)off) incl += v;
        }
        if (lane == 31) s_wsum[wid] = incl;
        __syncthreads();
        uint32_t before = incl - sum;
#pragma unroll
        for (unsigned v = 0; v < BK_WARPS; ++v) before += v < wid ? s_wsum[v] : 0u;
        for (uint32_t w = wlo; w < whi; ++w) {
            const uint32_t c = s_cnt[w];
            unsigned long long at = c ? atomicAdd(fill + w, (unsigned long long)c) : 0ull;
            if (at + c > cap) {  // the run does not fit: drop it, the chunk is filed again
                *overflow = 1;
                at = ~0ull;
            } else {
                at += (unsigned long long)w * cap;
            }
            s_dst[w] = at;
            s_off[w] = before;
            s_cnt[w] = before;
            before += c;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < KT; ++u)
            if ((have >> u) & 1u)
                bk_records<RT, ETA, M32>(ix, hp, wm, y[u], cell[u],
                               [&](uint32_t win, uint32_t at) { s_srt[atomicAdd(&s_cnt[win], 1u)] = at; });
        __syncthreads();
        // the runs, `run` lanes each (s_cnt is now each run's end)
        const uint32_t sub = threadIdx.x & (run - 1);
        for (uint32_t w = threadIdx.x / run; w < n_win; w += BK_THREADS / run) {
            const uint32_t lo = s_off[w], hi = s_cnt[w];
            const unsigned long long to = s_dst[w];
            if (to == ~0ull) continue;
            for (uint32_t i = lo + sub; i < hi; i += run) rec[to + (i - lo)] = s_srt[i];
        }
        __syncthreads();  // records and counters are rewritten by the next step
    }
}

// Apply window `win`: OR its bucket's records into the rows.  Where a word is
// hit over and over (a term that most documents hold puts two fifths of its
// row's window into ten words), atomics to it queue up one behind the other.
// With REPEATS (keys, which may be terms; not the windows of DNA), a block
// whose first records show that reads each word first and leaves it alone when
// the bit is set.  Elsewhere that read only adds traffic: 2e9 k-mers took 299
// ms instead of 137 with it, 5.5e7 terms over 1e5 documents 45 instead of 195.
template <bool REPEATS>
__global__ void __launch_bounds__(BK_APPLY_THREADS) k_bucket_apply(uint32_t* __restrict__ rows, uint64_t win_word0,
                                                                   const uint32_t* __restrict__ rec,
                                                                   const unsigned long long* __restrict__ fill,
                                                                   uint32_t win, uint64_t cap) {
    const uint64_t n = min((unsigned long long)cap, fill[win]);
    const uint32_t* r = rec + (uint64_t)win * cap;
    uint32_t* base = rows + win_word0;
    const uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, stride = (uint64_t)gridDim.x * blockDim.x;
    bool hot = false;
    if constexpr (REPEATS) {
        const uint32_t word = i0 < n ? r[i0] >> 5 : ~0u - threadIdx.x;  // (beyond the bucket: all different)
        hot = __syncthreads_or(__popc(__match_any_sync(FULL, word)) >= 2);
    }
    for (uint64_t i = i0; i < n; i += stride) {
        const uint32_t x = __ldcs(r + i);  // streamed once
        uint32_t* at = base + (x >> 5);
        const uint32_t bit = 1u << (x & 31);
        if (!REPEATS || !hot || !(__ldcg(at) & bit)) atomicOr(at, bit);
    }
}

using ScatterKernel = void (*)(IndexView, HashParams, BatchView, uint64_t, uint64_t, WindowMap, uint32_t, uint32_t,
                               uint64_t, uint32_t*, unsigned long long*, unsigned long long*, const DevStatus*);

// keys a thread takes per step: as many as its record slots hold
template <int ETA, bool M32>
static ScatterKernel scatter_kernel(uint32_t R, int kt) {
    if (R > 8) return kt >= 2 ? &k_bucket_scatter<16, 2, ETA, M32> : &k_bucket_scatter<16, 1, ETA, M32>;
    return kt >= 4   ? &k_bucket_scatter<8, 4, ETA, M32>
           : kt >= 2 ? &k_bucket_scatter<8, 2, ETA, M32>
                     : &k_bucket_scatter<8, 1, ETA, M32>;
}

cudaError_t launch_bucket_scatter(const IndexView& ix, const HashParams& hp, const BatchView& b, uint64_t p_lo,
                                  uint64_t p_hi, uint64_t rows_per_win, uint32_t n_win, uint64_t cap, uint32_t* rec,
                                  unsigned long long* fill, unsigned long long* overflow, const DevStatus* st,
                                  int num_sms, cudaStream_t s) {
    if (p_hi <= p_lo) return cudaSuccess;
    if (n_win > BK_MAX_WINDOWS || ix.R * ix.eta > BK_SLOTS) return cudaErrorInvalidValue;
    WindowMap wm{rows_per_win, 0, 0};
    const uint64_t rows_total = (uint64_t)ix.R * ix.m;
    while (wm.unit < 16 && !((rows_per_win >> wm.unit) & 1)) ++wm.unit;
    const uint64_t d = rows_per_win >> wm.unit;
    if (rows_total <= (1ull << 32) && d > 1 && ((rows_total - 1) >> wm.unit) * d < (1ull << 32))
        wm.magic = (uint32_t)(((1ull << 32) + d - 1) / d);
    const uint32_t fit = BK_SLOTS / (ix.R * ix.eta);
    const int kt = ix.R > 8 ? (fit >= 2 ? 2 : 1) : fit >= 4 ? 4 : fit >= 2 ? 2 : 1;
    const uint64_t span = (uint64_t)kt * BK_THREADS;
    const ScatterKernel f = !wm.magic      ? scatter_kernel<EMAX, false>(ix.R, kt)
                            : ix.eta == 1 ? scatter_kernel<1, true>(ix.R, kt)
                            : ix.eta == 2 ? scatter_kernel<2, true>(ix.R, kt)
                            : ix.eta == 3 ? scatter_kernel<3, true>(ix.R, kt)
                                          : scatter_kernel<4, true>(ix.R, kt);
    // records by window, then destination, count and offset of every window
    const size_t smem = (size_t)BK_TILE_RECORDS * 4 + (size_t)n_win * 16;
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    uint64_t blocks = (p_hi - p_lo + span - 1) / span;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, BK_THREADS, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const uint64_t most = (uint64_t)num_sms * per_sm;
    if (blocks > most) blocks = most;
    // lanes a run, near its mean length
    uint32_t run = 32;
    while (run > 4 && (uint64_t)run * n_win > span * ix.R * ix.eta) run /= 2;
    f<<<(unsigned)blocks, BK_THREADS, smem, s>>>(ix, hp, b, p_lo, p_hi, wm, n_win, run, cap, rec, fill, overflow, st);
    return cudaGetLastError();
}

cudaError_t launch_bucket_apply(uint32_t* rows, uint64_t win_word0, const uint32_t* rec,
                                const unsigned long long* fill, uint32_t win, uint64_t cap, bool repeats, int num_sms,
                                cudaStream_t s) {
    const auto f = repeats ? &k_bucket_apply<true> : &k_bucket_apply<false>;
    f<<<(unsigned)(num_sms * 8), BK_APPLY_THREADS, 0, s>>>(rows, win_word0, rec, fill, win, cap);
    return cudaGetLastError();
}

}  // namespace rgb
