// k_query_wide.cu -- the batched RAMBO query (Algorithm 2, Sec. 3.2, with the
// sequence rule of Sec. 3.2.1) for indexes whose rows are too wide, or whose
// tables too many, for the register-tiled kernel: the paper's stacked
// whole-genome index (B = 50000, R = 5, folded to 25000 / 12500 / 6250;
// Sec. 5.2) and its ClueWeb09 index (B = 2e4, R = 4; Sec. 5.3) have rows of
// 2.5-6.25 KB.
//
// One thread block answers one query at a time, taking query indices from
// the same device work queue (atomic ticket) as the other kernel.  The
// query's per-table cell masks M_r (B bits each) live in shared memory.
// Terms are taken QW_TERMS at a time: every thread takes columns of four words
// of a table (16-byte loads, coalesced across the block) and ANDs the R * eta
// rows of the step's terms into the masks, all of a column's loads in flight
// together.  After each step the block checks whether some table's mask is
// empty (then no set can hold every term: the first FALSE is conclusive,
// Sec. 3.2.1) and stops.
//
// With o.dmask set, a surviving query is handed over as its masks and the set
// kernel (k_query_set.cu) does the rest; otherwise the block does:
// Set stage: every registered ID i is tested against bit phi_r(i) of M_r for
// every table (the union over hit cells per table and the intersection
// across tables of Algorithm 2); the survivors are counted, a range of the
// staging arena is reserved, and a second pass writes them in ascending
// order with a block-wide ordered compaction.
#include "rambo_impl.cuh"

namespace rgb {

constexpr int QW_TERMS = 4;  // terms per step

// shared memory: masks [R][S] words, then the step's hashed keys, then control words
size_t query_wide_smem_bytes(uint32_t R, uint32_t S) {
    return (((size_t)R * S * 4 + 15) & ~(size_t)15) + QW_TERMS * 8 + 64 * 4;
}

// VW words of a row (S a multiple of VW)
template <int VW>
__device__ __forceinline__ void qw_load(const uint32_t* p, uint32_t (&v)[VW]) {
    if constexpr (VW == 1) {
        v[0] = __ldg(p);
    } else if constexpr (VW == 2) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(p));
        v[0] = x.x, v[1] = x.y;
    } else {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p));
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    }
}

// ANDs the rows of the step's terms (bit u of `terms`: term u is there, its
// hash in y[u]) into the masks and returns the tables this thread saw a set
// bit in.  `first`: the masks hold nothing yet.
template <int VW, int ETA>
__device__ __forceinline__ uint32_t qw_step(const IndexView& ix, const HashParams& hp, const uint64_t* y,
                                            uint32_t terms, bool first, uint32_t* sM) {
    const uint32_t cpt = ix.S / VW, cols = ix.R * cpt;  // columns of a table, of all
    uint32_t nz = 0;
    for (uint32_t f = threadIdx.x; f < cols; f += QW_THREADS) {
        const uint32_t r = f / cpt, w = (f - r * cpt) * VW;
        const uint32_t* base = ix.rows + (uint64_t)r * ix.m * ix.S + w;
        uint32_t v[QW_TERMS][ETA][VW];
#pragma unroll
        for (int u = 0; u < QW_TERMS; ++u)
#pragma unroll
            for (int j = 0; j < ETA; ++j)
                if (((terms >> u) & 1u) && j < (int)ix.eta)
                    qw_load<VW>(base + ((hp.s[r][j] * y[u]) >> ix.shift) * ix.S, v[u][j]);
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < VW; ++i) {
            uint32_t x = first ? ~0u : sM[r * ix.S + w + i];
#pragma unroll
            for (int u = 0; u < QW_TERMS; ++u)
#pragma unroll
                for (int j = 0; j < ETA; ++j)
                    if (((terms >> u) & 1u) && j < (int)ix.eta) x &= v[u][j][i];
            sM[r * ix.S + w + i] = x;
            any |= x;
        }
        if (any) nz |= 1u << r;
    }
    return nz;
}

template <int VW, int ETA>
__global__ void __launch_bounds__(QW_THREADS) k_query_wide(IndexView ix, HashParams hp, BatchView b, QueryOut o,
                                                           DevStatus* st) {
    extern __shared__ __align__(16) unsigned char qw_smem[];
    const uint32_t R = ix.R, S = ix.S, eta = ix.eta;
    uint32_t* sM = reinterpret_cast<uint32_t*>(qw_smem);                             // [R][S]
    uint64_t* sY = reinterpret_cast<uint64_t*>(qw_smem + (((size_t)R * S * 4 + 15) & ~(size_t)15));  // [QW_TERMS]
    uint32_t* ctl = reinterpret_cast<uint32_t*>(sY + QW_TERMS);                      // control
    unsigned long long* ctl_q = reinterpret_cast<unsigned long long*>(ctl);         // [0..1] ticket
    unsigned long long* ctl_start = reinterpret_cast<unsigned long long*>(ctl + 2); // [2..3] staging start or slot
    uint32_t* ctl_nz = ctl + 4;                                                      // [4] tables still non-empty
    uint32_t* ctl_act = ctl + 5;                                                     // [5] the step's terms
    uint32_t* warp_cnt = ctl + 16;                                                   // [16..23] per-warp counts

    bv_resolve(b);
    if (query_batch_rejected(b, st)) return;
    const unsigned tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    constexpr unsigned nthreads = QW_THREADS, nwarps = nthreads >> 5;
    const uint32_t rmask = R >= 32 ? ~0u : ((1u << R) - 1u);
    unsigned long long probed = 0, rows_read = 0;

    for (;;) {
        if (tid == 0) *ctl_q = atomicAdd(&st->ticket, 1ull);
        __syncthreads();
        const unsigned long long t = *ctl_q;
        if (t >= b.n) break;
        const unsigned long long q = b.perm ? (unsigned long long)__ldg(b.perm + t) : t;
        const uint64_t a = __ldg(b.offsets + q) - b.off0;
        const uint64_t e = __ldg(b.offsets + q + 1) - b.off0;
        const uint64_t nkeys = b.seq ? (e - a - b.k + 1) : (e - a);  // >= 1 (validated)

        bool alive = true;
        // Steps visit terms in a strided order: step s takes terms s, s +
        // nsteps, s + 2 nsteps, ... so the first steps sample the whole query
        // (a substitution makes k consecutive windows absent).
        const uint64_t nsteps = (nkeys + QW_TERMS - 1) / QW_TERMS;
        for (uint64_t s = 0; s < nsteps && alive; ++s) {
            if (wid == 0) {
                // this step's terms, a lane each
                const uint64_t idx = s + (uint64_t)lane * nsteps;
                bool act = lane < QW_TERMS && idx < nkeys;
                uint64_t key = 0;
                if (act) {
                    if (b.seq) {
                        act = !b.skipn || window_resolved(b.nmask, a + idx, b.k);
                        key = kmer_at(b.packed, a + idx, b.k);
                        if (b.canon) key = canonical_kmer(key, b.k);
                    } else {
                        key = __ldg(b.keys + a + idx);
                    }
                }
                if (lane < QW_TERMS) sY[lane] = mix64(key);
                const unsigned terms = __ballot_sync(FULL, act);
                if (lane == 0) {
                    *ctl_act = terms;
                    *ctl_nz = 0;
                }
            }
            __syncthreads();
            const uint32_t terms = *ctl_act;
            const unsigned nact = __popc(terms);
            uint32_t nz = qw_step<VW, ETA>(ix, hp, sY, terms, s == 0, sM);
            // tables with a set bit anywhere (R <= 16 fits one word)
            nz = __reduce_or_sync(FULL, nz);
            if (lane == 0 && nz) atomicOr(ctl_nz, nz);
            __syncthreads();
            probed += nact;
            rows_read += (unsigned long long)nact * R * eta;
            if ((*ctl_nz & rmask) != rmask) alive = false;
            __syncthreads();  // ctl words are rewritten by the next step
        }
        if (o.dmask) {
            if (tid == 0) {
                o.qcount[q] = 0;
                if (alive) *ctl_start = atomicAdd(&st->n_handed, 1ull);
            }
            if (!alive) continue;  // (the ticket is rewritten, and read behind the next barrier)
            __syncthreads();
            const uint64_t slot = *ctl_start;
            for (uint32_t w = tid; w < R * S; w += nthreads) o.dmask[slot * (R * S) + w] = sM[w];
            if (tid == 0) {
                o.dq[slot] = (uint32_t)q;
                o.qstart[q] = slot * set_pitch(ix.K) | QSTART_BITMAP;
            }
            __syncthreads();  // masks and control words are reused by the next query
            continue;
        }

        uint32_t count = 0;
        unsigned long long start = 0;
        if (alive) {
            // pass 1: count the registered sets hit in every table
            for (uint64_t i0 = 0; i0 < ix.K; i0 += nthreads) {
                const uint64_t i = i0 + tid;
                bool ok = i < ix.K && ((__ldg(ix.reg + (i >> 5)) >> (i & 31)) & 1u);
                if (ok) {
                    const uint16_t* ph = ix.phi + i * ix.ps;
                    for (uint32_t r = 0; r < R && ok; ++r) {
                        const uint32_t c = __ldg(ph + r);
                        ok = (sM[r * S + (c >> 5)] >> (c & 31)) & 1u;
                    }
                }
                count += (uint32_t)__syncthreads_count(ok);
            }
            if (tid == 0 && count) *ctl_start = atomicAdd(&st->cursor, (unsigned long long)count);
            __syncthreads();
            start = count ? *ctl_start : 0ull;
            if (count && start + count <= o.stage_cap) {
                // pass 2: the same test, survivors written in ascending order
                uint32_t at = 0;
                for (uint64_t i0 = 0; i0 < ix.K; i0 += nthreads) {
                    const uint64_t i = i0 + tid;
                    bool ok = i < ix.K && ((__ldg(ix.reg + (i >> 5)) >> (i & 31)) & 1u);
                    if (ok) {
                        const uint16_t* ph = ix.phi + i * ix.ps;
                        for (uint32_t r = 0; r < R && ok; ++r) {
                            const uint32_t c = __ldg(ph + r);
                            ok = (sM[r * S + (c >> 5)] >> (c & 31)) & 1u;
                        }
                    }
                    const unsigned bal = __ballot_sync(0xffffffffu, ok);
                    if (lane == 0) warp_cnt[wid] = __popc(bal);
                    __syncthreads();
                    uint32_t before = 0, total = 0;
                    for (unsigned v = 0; v < nwarps; ++v) {
                        const uint32_t c = warp_cnt[v];
                        if (v < wid) before += c;
                        total += c;
                    }
                    if (ok) o.stage[start + at + before + __popc(bal & ((1u << lane) - 1u))] = (uint32_t)i;
                    at += total;
                    __syncthreads();  // warp counts are rewritten by the next chunk
                }
            }
        }
        if (tid == 0) {
            o.qcount[q] = count;
            o.qstart[q] = start;
        }
        __syncthreads();  // masks and control words are reused by the next query
    }
    if (tid == 0 && probed) atomicAdd(&st->keys_probed, probed);
    if (tid == 0 && rows_read) atomicAdd(&st->rows_read, rows_read);
}

using WideKernel = void (*)(IndexView, HashParams, BatchView, QueryOut, DevStatus*);

// column width by the row stride (1, 2 or a multiple of 4 words), and eta
static WideKernel wide_kernel(uint32_t S, uint32_t eta) {
    if (S == 1) return eta <= 2 ? &k_query_wide<1, 2> : &k_query_wide<1, 4>;
    if (S == 2) return eta <= 2 ? &k_query_wide<2, 2> : &k_query_wide<2, 4>;
    return eta <= 2 ? &k_query_wide<4, 2> : &k_query_wide<4, 4>;
}

int query_wide_blocks_per_sm(uint32_t R, uint32_t S, uint32_t eta) {
    const size_t smem = query_wide_smem_bytes(R, S);
    const WideKernel f = wide_kernel(S, eta);
    if (smem > 48 * 1024 && cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, QW_THREADS, smem) != cudaSuccess) return 0;
    return nb;
}

cudaError_t launch_query_wide(const IndexView& ix, const HashParams& hp, const BatchView& b, const QueryOut& o,
                              int blocks, DevStatus* st, cudaStream_t s) {
    if (b.n == 0 && !b.desc) return cudaSuccess;
    const size_t smem = query_wide_smem_bytes(ix.R, ix.S);
    const WideKernel f = wide_kernel(ix.S, ix.eta);
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    f<<<(unsigned)(blocks > 0 ? blocks : 1), QW_THREADS, smem, s>>>(ix, hp, b, o, st);
    return cudaGetLastError();
}

cudaError_t load_query_wide_kernel() {
    for (const uint32_t S : {1u, 2u, 4u})
        for (const uint32_t eta : {2u, 4u}) {
            cudaFuncAttributes a;
            const cudaError_t e = cudaFuncGetAttributes(&a, wide_kernel(S, eta));
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace rgb
