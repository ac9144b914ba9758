// k_probe.cuh -- the probes of Algorithm 2 (Sec. 3.2, with the sequence rule
// of Sec. 3.2.1) for batches whose set stage the set kernel runs
// (k_query_set.cu).  Steps A1-A4 are those of k_query.cuh; a query whose R
// per-table cell masks all keep a hit cell is handed over as those masks.
//
// Without a set stage a warp needs no shared-memory bitmap of the ID space and
// nothing holds it up between a query's rows and the next query's.  What
// bounds it: the rate of isolated DRAM accesses for long queries (1e6 uneven
// sequences, 7.2e8 rows: 15.4 ms with the set stage in the same kernel, 14.15
// here; 2e5 short reads 4.77 -> 3.96), latency for short ones, which therefore
// go 32 / G to a warp (1e5 document queries 0.26 ms, 1e4 single k-mers 33 us by
// warps, 8 by lane groups).
//
// Three instances, picked by the batch's mean number of terms and its size
// (probe_short, qk_group_size); a launch whose instance is not the batch's
// returns at once, so a captured graph holds them and the batch, read on the
// device, picks:
//   PB_LANES   up to PB_SHORT_MEAN terms a query, PB_MANY queries or more:
//              each group of G lanes answers a query of its own, one term a
//              step, so a warp has 32 / G queries in flight and nothing to
//              reduce across terms.  Queries of such a batch with more than
//              PB_SHORT_MOST terms are listed for PB_WARP;
//   PB_WARP    a warp per query, 32 / G terms a step;
//   PB_GROUP   longer queries, too few to fill the grid: P warps of a block
//              share one.
// Batches of fewer than PB_MANY queries wait for latency, not for bandwidth:
// they read every table of the first step at once instead of screening on
// table 0.
#pragma once

#include "k_query.cuh"

namespace rgb {

constexpr uint64_t PB_MANY = 2048;
constexpr uint64_t PB_SHORT_MEAN = 8;   // mean terms a query up to which lane groups answer them
constexpr uint64_t PB_SHORT_MOST = 32;  // longer ones of such a batch take a whole warp

// Tables whose rows a lane group has in flight: up to 32 registers of them.
template <int V, int ETA>
constexpr int PB_TABLES = ETA * V >= 16 ? 2 : ETA * V >= 8 ? 4 : 8;

// Up to PB_SHORT_MEAN terms a query on average (unless a group size was asked for).
__host__ __device__ inline bool probe_short(uint64_t n, uint64_t total, int seq, uint32_t k, int group) {
    const uint64_t cut = seq ? n * (uint64_t)(k - 1) : 0;
    return group <= 1 && total <= cut + PB_SHORT_MEAN * n;
}

// The instance that serves a batch (P: its warps per query; wpb and
// group_warps: of PB_GROUP's launch, whose blocks may be wider than the others').
__host__ __device__ inline int probe_mode(const BatchView& b, int group, unsigned wpb, uint64_t group_warps, int lanes,
                                          unsigned& P) {
    P = 1;
    if (probe_short(b.n, b.total, b.seq, b.k, group)) return lanes && b.n >= PB_MANY ? PB_LANES : PB_WARP;
    P = qk_group_size(b.n, group, wpb, group_warps, 1);
    return P > 1 ? PB_GROUP : PB_WARP;
}

// Row reads use the default cache operator alone (read-only path, no L1
// allocation, 64-byte L2 fetch; row_load 7): a switch over the eight of them
// at each of a step's R * eta reads made the kernel spill.  What spills all
// the same, at 128 registers: instances of V = 4 and eta <= 2 (8 to 64 bytes;
// 44 in <4, 1, 2, PB_WARP>, rows of 16 bytes) and the lane groups of eta > 2
// (40 to 120).
template <int V>
__device__ __forceinline__ void probe_load(const uint32_t* p, uint32_t (&v)[V]) {
    if constexpr (V == 1)
        asm volatile("ld.global.nc.L1::no_allocate.L2::64B.u32 %0, [%1];" : "=r"(v[0]) : "l"(p));
    else if constexpr (V == 2)
        asm volatile("ld.global.nc.L1::no_allocate.L2::64B.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "l"(p));
    else
        asm volatile("ld.global.nc.L1::no_allocate.L2::64B.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                     : "l"(p));
}

// Reads the eta rows of tables [rlo, rhi) at the key hashed to y, TC tables
// (all of their rows before any is used) at a time, and gives `take` each
// table's AND of them word by word (~0 in a lane that reads nothing).
template <int V, int ETA, int TC, class F>
__device__ __forceinline__ void probe_rows(const IndexView& ix, const HashParams& hp, uint64_t y, bool ld, int rlo,
                                           int rhi, uint32_t w0, F take) {
    const int eta = (int)ix.eta;
#pragma unroll
    for (int r0 = 0; r0 < RF; r0 += TC) {
        uint32_t val[TC][ETA][V];
#pragma unroll
        for (int u = 0; u < TC; ++u) {
            const int r = r0 + u;
            if (r >= rlo && r < rhi && ld) {
                const uint32_t* rb = ix.rows + (uint64_t)r * ix.m * ix.S + w0;
#pragma unroll
                for (int j = 0; j < ETA; ++j) {
                    if (j < eta) {
                        const uint64_t pos = (hp.s[r][j] * y) >> ix.shift;
                        probe_load<V>(rb + pos * ix.S, val[u][j]);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < TC; ++u) {
            const int r = r0 + u;
            if (r >= rlo && r < rhi) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    uint32_t x = ~0u;
                    if (ld) {
#pragma unroll
                        for (int j = 0; j < ETA; ++j)
                            if (j < eta) x &= val[u][j][v];
                    }
                    take(r, v, x);
                }
            }
        }
    }
}

__device__ __forceinline__ uint64_t probe_key(const BatchView& b, uint64_t p) {
    if (!b.seq) return __ldg(b.keys + p);
    const uint64_t key = kmer_at(b.packed, p, b.k);
    return b.canon ? canonical_kmer(key, b.k) : key;
}

template <int V>
__device__ __forceinline__ void store_words(uint32_t* p, const uint32_t (&v)[V]) {
    if constexpr (V == 1) *p = v[0];
    else if constexpr (V == 2) *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
    else *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
}

// Hands query q over in slot `slot`: this lane's words of its masks, and (lead) where its answer goes.
template <int V>
__device__ __forceinline__ void hand_over(const IndexView& ix, const QueryOut& o, uint64_t q, uint64_t slot,
                                          const uint32_t (&M)[RF][V], uint32_t w0, bool has_words, bool lead) {
    uint32_t* m = o.dmask + slot * (ix.R * ix.S) + w0;
#pragma unroll
    for (int r = 0; r < RF; ++r)
        if (r < (int)ix.R && has_words) store_words<V>(m + r * ix.S, M[r]);
    if (lead) {
        o.dq[slot] = (uint32_t)q;
        o.qstart[q] = slot * set_pitch(ix.K) | QSTART_BITMAP;
    }
}

// The tables of M that keep a hit cell in this lane's words.
template <int V>
__device__ __forceinline__ uint32_t nonempty(const IndexView& ix, const uint32_t (&M)[RF][V]) {
    uint32_t nz = 0;
#pragma unroll
    for (int r = 0; r < RF; ++r) {
        if (r < (int)ix.R) {
            uint32_t any = 0;
#pragma unroll
            for (int v = 0; v < V; ++v) any |= M[r][v];
            if (any) nz |= 1u << r;
        }
    }
    return nz;
}

// One query by the whole warp; true (and its masks in M, in every lane group)
// when it survives.  Step s visits terms s*KPS + g (input order) or
// g*nsteps + s (strided: the first step samples the whole query evenly); with
// screening (order 2) the first step reads table 0 alone, then the others.
template <int V, int G, int ETA>
__device__ __forceinline__ bool probe_warp(const IndexView& ix, const HashParams& hp, const BatchView& b, uint64_t a,
                                           uint64_t nkeys, int order, uint32_t w0, bool has_words,
                                           uint32_t (&M)[RF][V], unsigned long long& probed,
                                           unsigned long long& rows_read) {
    constexpr int KPS = 32 / G;
    const unsigned lane = threadIdx.x & 31, grp = lane / G, slot = lane % G;
    const int R = (int)ix.R;
    const uint32_t rmask = (1u << R) - 1u;
#pragma unroll
    for (int r = 0; r < RF; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) M[r][v] = has_words ? ~0u : 0u;
    const uint64_t nsteps = (nkeys + KPS - 1) / KPS;
    const bool screen = order >= 2 && R > 1;
    const uint64_t nphases = nsteps + (screen ? 1 : 0);
#pragma unroll 1
    for (uint64_t ph = 0; ph < nphases; ++ph) {
        const uint64_t s = screen ? (ph == 0 ? 0 : ph - 1) : ph;
        const int rlo = (screen && ph == 1) ? 1 : 0;
        const int rhi = (screen && ph == 0) ? 1 : R;
        const uint64_t idx = order ? (uint64_t)grp * nsteps + s : s * KPS + grp;
        // skip-N: a window holding an unresolved base is not a term
        const bool act = idx < nkeys && (!b.skipn || window_resolved(b.nmask, a + idx, b.k));
        const uint64_t y = mix64(act ? probe_key(b, a + idx) : 0);
        probe_rows<V, ETA, RF>(ix, hp, y, act && has_words, rlo, rhi, w0,
                            [&](int r, int v, uint32_t x) { M[r][v] &= qk_and_groups<G>(x); });
        const uint32_t nz = __reduce_or_sync(FULL, nonempty<V>(ix, M));
        const unsigned nact = __popc(__ballot_sync(FULL, act && slot == 0));
        if (!(screen && ph == 1)) probed += nact;  // the screened terms were counted in phase 0
        rows_read += (unsigned long long)nact * (unsigned)(rhi - rlo) * ix.eta;
        if (nz != rmask) return false;
    }
    return true;
}

// One query by this lane group (32 / G queries a warp; warp-uniform call), the
// group's masks in M; `alive` says whether there is one, and returns whether
// it survived.
template <int V, int G, int ETA>
__device__ __forceinline__ bool probe_group(const IndexView& ix, const HashParams& hp, const BatchView& b, uint64_t a,
                                            uint64_t nkeys, bool alive, int order, uint32_t w0,
                                            bool has_words, uint32_t (&M)[RF][V], unsigned long long& probed,
                                            unsigned long long& rows_read) {
    const unsigned slot = (threadIdx.x & 31) % G;
    const int R = (int)ix.R;
    const uint32_t rmask = (1u << R) - 1u;
    const bool screen = order >= 2 && R > 1;
#pragma unroll
    for (int r = 0; r < RF; ++r)
#pragma unroll
        for (int v = 0; v < V; ++v) M[r][v] = has_words ? ~0u : 0u;
#pragma unroll 1
    for (uint64_t t = 0; __any_sync(FULL, alive && t < nkeys); ++t) {
        const bool act = alive && t < nkeys && (!b.skipn || window_resolved(b.nmask, a + t, b.k));
        const uint64_t y = mix64(act ? probe_key(b, a + t) : 0);
        const int phases = screen && t == 0 ? 2 : 1;
#pragma unroll 1
        for (int ph = 0; ph < phases; ++ph) {
            const int rlo = phases == 2 && ph == 1 ? 1 : 0;
            const int rhi = phases == 2 && ph == 0 ? 1 : R;
            const bool go = act && alive;
            probe_rows<V, ETA, PB_TABLES<V, ETA>>(ix, hp, y, go && has_words, rlo, rhi, w0,
                                [&](int r, int v, uint32_t x) { M[r][v] &= x; });
            uint32_t nz = nonempty<V>(ix, M);
#pragma unroll
            for (int off = 1; off < G; off <<= 1) nz |= __shfl_xor_sync(FULL, nz, off);
            const unsigned nact = __popc(__ballot_sync(FULL, go && slot == 0));
            if (ph == 0) probed += nact;
            rows_read += (unsigned long long)nact * (unsigned)(rhi - rlo) * ix.eta;
            alive = alive && nz == rmask;
        }
    }
    return alive;
}

template <int V, int G, int ETA, int MODE>
__global__ void __launch_bounds__(QK_THREADS_MAX, RF * ETA * V <= 64 ? 2 : 1)
    k_probe(IndexView ix, HashParams hp, BatchView b, QueryOut o, int batch, int order, int group, int group_wpb,
            unsigned long long group_warps, int lanes, DevStatus* st) {
    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned grp = lane / G, slot = lane % G;
    const uint32_t w0 = slot * V;
    const bool has_words = w0 < ix.S;
    bv_resolve(b);
    if (query_batch_rejected(b, st)) return;
    unsigned P;
    const int mode = probe_mode(b, group, (unsigned)group_wpb, group_warps, lanes, P);
    const bool listed = MODE == PB_WARP && mode == PB_LANES;  // the long queries that lane groups listed
    if (mode != MODE && !listed) return;
    if (b.n < PB_MANY && order == 2) order = 1;
    unsigned long long probed = 0, rows_read = 0;
    uint32_t M[RF][V];
    // a warp's first queries need no ticket; the work queue hands out the rest
    const unsigned long long warp = blockIdx.x * (unsigned long long)(blockDim.x >> 5) + wid;
    auto next = [&](unsigned long long* ticket, unsigned take) {
        unsigned long long q = 0;
        if (lane == 0) q = atomicAdd(ticket, (unsigned long long)take) + gridDim.x * (unsigned long long)(blockDim.x >> 5) * take;
        return __shfl_sync(FULL, q, 0);
    };
    if constexpr (MODE == PB_LANES) {
        constexpr unsigned PER = 32 / G;  // queries a warp has in flight
        for (unsigned long long q0 = warp * PER; q0 < b.n; q0 = next(&st->ticket, PER)) {
            const uint64_t t = q0 + grp;
            bool have = t < b.n;
            uint64_t q = 0, a = 0, nkeys = 0;
            if (have) {
                q = b.perm ? (uint64_t)__ldg(b.perm + t) : t;
                a = __ldg(b.offsets + q) - b.off0;
                nkeys = __ldg(b.offsets + q + 1) - b.off0 - a;
                if (b.seq) nkeys -= b.k - 1;
                if (nkeys > PB_SHORT_MOST) {
                    have = false;
                    if (slot == 0) o.dlong[atomicAdd(&st->n_long, 1ull)] = (uint32_t)q;
                } else if (slot == 0) {
                    o.qcount[q] = 0;
                }
            }
            const bool alive =
                probe_group<V, G, ETA>(ix, hp, b, a, nkeys, have, order, w0, has_words, M, probed, rows_read);
            const unsigned won = __ballot_sync(FULL, alive && slot == 0);
            unsigned long long s0 = 0;
            if (won && lane == 0) s0 = atomicAdd(&st->n_handed, (unsigned long long)__popc(won));
            s0 = __shfl_sync(FULL, s0, 0);
            if (alive)
                hand_over<V>(ix, o, q, s0 + __popc(won & ((1u << (lane - slot)) - 1u)), M, w0, has_words, slot == 0);
        }
    } else if constexpr (MODE == PB_WARP) {
        const uint64_t n = listed ? st->n_long : b.n;
        unsigned long long* ticket = listed ? &st->ticket_long : &st->ticket;
        for (unsigned long long q0 = warp * batch; q0 < n; q0 = next(ticket, batch)) {
            const unsigned long long q1 = min(q0 + (unsigned long long)batch, (unsigned long long)n);
            for (unsigned long long t = q0; t < q1; ++t) {
                const uint64_t q = listed ? (uint64_t)o.dlong[t] : b.perm ? (uint64_t)__ldg(b.perm + t) : t;
                const uint64_t a = __ldg(b.offsets + q) - b.off0;
                uint64_t nkeys = __ldg(b.offsets + q + 1) - b.off0 - a;
                if (b.seq) nkeys -= b.k - 1;
                const bool alive =
                    probe_warp<V, G, ETA>(ix, hp, b, a, nkeys, order, w0, has_words, M, probed, rows_read);
                if (lane == 0) o.qcount[q] = 0;
                if (!alive) continue;
                unsigned long long s0 = 0;
                if (lane == 0) s0 = atomicAdd(&st->n_handed, 1ull);
                s0 = __shfl_sync(FULL, s0, 0);
                hand_over<V>(ix, o, q, s0, M, w0, has_words && grp == 0, lane == 0);
            }
        }
    } else {
        // the group's shared state: [QK_CTL] control words, then [R][S] masks
        extern __shared__ uint32_t pb_smem[];
        const unsigned gi = wid / P, gw = wid % P;
        const bool leader = gw == 0 && lane == 0;
        const uint32_t words = ix.R * ix.S;
        uint32_t* ctl = pb_smem + gi * ((QK_CTL + words + 3u) & ~3u);
        uint32_t* sM = ctl + QK_CTL;
        volatile unsigned long long* ctl_ticket = reinterpret_cast<volatile unsigned long long*>(ctl);
        volatile uint32_t* ctl_dead = ctl + 2;
        constexpr int KPS = 32 / G;
        const int R = (int)ix.R;
        const uint32_t rmask = (1u << R) - 1u;
        const bool screen = order >= 2 && R > 1;
        for (;;) {
            if (leader) {
                *ctl_ticket = atomicAdd(&st->ticket, 1ull);
                *ctl_dead = 0;
            }
            for (uint32_t w = gw * 32 + lane; w < words; w += P * 32) sM[w] = ~0u;
            qk_group_sync(P, gi);
            const unsigned long long t = *ctl_ticket;
            if (t >= b.n) break;
            const uint64_t q = b.perm ? (uint64_t)__ldg(b.perm + t) : t;
            const uint64_t a = __ldg(b.offsets + q) - b.off0;
            uint64_t nkeys = __ldg(b.offsets + q + 1) - b.off0 - a;
            if (b.seq) nkeys -= b.k - 1;
#pragma unroll
            for (int r = 0; r < RF; ++r)
#pragma unroll
                for (int v = 0; v < V; ++v) M[r][v] = has_words ? ~0u : 0u;
            // warp gw takes steps gw, gw + P, ... (see probe_warp)
            const uint64_t nsteps = (nkeys + KPS - 1) / KPS;
            const uint64_t mine = nsteps > gw ? (nsteps - gw + P - 1) / P : 0;
            const uint64_t nphases = mine + ((screen && mine) ? 1 : 0);
            bool alive = true;
#pragma unroll 1
            for (uint64_t ph = 0; ph < nphases; ++ph) {
                if (__shfl_sync(FULL, *ctl_dead, 0)) break;  // another warp found an empty table
                const uint64_t s = gw + (uint64_t)P * (screen ? (ph == 0 ? 0 : ph - 1) : ph);
                const int rlo = (screen && ph == 1) ? 1 : 0;
                const int rhi = (screen && ph == 0) ? 1 : R;
                const uint64_t idx = order ? (uint64_t)grp * nsteps + s : s * KPS + grp;
                const bool act = idx < nkeys && (!b.skipn || window_resolved(b.nmask, a + idx, b.k));
                const uint64_t y = mix64(act ? probe_key(b, a + idx) : 0);
                probe_rows<V, ETA, RF>(ix, hp, y, act && has_words, rlo, rhi, w0,
                                    [&](int r, int v, uint32_t x) { M[r][v] &= qk_and_groups<G>(x); });
                const uint32_t nz = __reduce_or_sync(FULL, nonempty<V>(ix, M));
                const unsigned nact = __popc(__ballot_sync(FULL, act && slot == 0));
                if (!(screen && ph == 1)) probed += nact;
                rows_read += (unsigned long long)nact * (unsigned)(rhi - rlo) * ix.eta;
                if (nz != rmask) {
                    alive = false;
                    if (lane == 0) *ctl_dead = 1;
                    break;
                }
            }
            // AND of the warps' partial masks (one that stopped early holds a superset)
            if (alive && mine && grp == 0 && has_words) {
#pragma unroll
                for (int r = 0; r < RF; ++r)
                    if (r < R)
#pragma unroll
                        for (int v = 0; v < V; ++v) atomicAnd(sM + r * ix.S + w0 + v, M[r][v]);
            }
            qk_group_sync(P, gi);
            if (gw == 0) {
                bool survives = *ctl_dead == 0;
                for (int r = 0; r < R && survives; ++r) {
                    uint32_t any = 0;
                    for (uint32_t w = lane; w < ix.S; w += 32) any |= sM[r * ix.S + w];
                    survives = __any_sync(FULL, any != 0);
                }
                if (lane == 0) o.qcount[q] = 0;
                if (survives) {
                    unsigned long long s0 = 0;
                    if (lane == 0) s0 = atomicAdd(&st->n_handed, 1ull);
                    s0 = __shfl_sync(FULL, s0, 0);
                    for (uint32_t w = lane; w < words; w += 32) o.dmask[s0 * words + w] = sM[w];
                    if (lane == 0) {
                        o.dq[s0] = (uint32_t)q;
                        o.qstart[q] = s0 * set_pitch(ix.K) | QSTART_BITMAP;
                    }
                }
            }
            qk_group_sync(P, gi);  // masks and control words are reused by the next query
        }
    }
    if (lane == 0 && probed) atomicAdd(&st->keys_probed, probed);
    if (lane == 0 && rows_read) atomicAdd(&st->rows_read, rows_read);
}

}  // namespace rgb
