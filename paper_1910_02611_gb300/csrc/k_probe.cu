// k_probe.cu -- dispatch of the probe kernel instances and occupancy helpers.
#include "k_probe.cuh"

namespace rgb {

using ProbeKernel = void (*)(IndexView, HashParams, BatchView, QueryOut, int, int, int, int, unsigned long long, int,
                             DevStatus*);
ProbeKernel probe_kernel_e2(int V, int G, int mode);
ProbeKernel probe_kernel_e4(int V, int G, int mode);

static ProbeKernel probe_kernel(int V, int G, uint32_t eta, int mode) {
    return eta <= 2 ? probe_kernel_e2(V, G, mode) : probe_kernel_e4(V, G, mode);
}

// Shared memory of the grouped instance: control words and masks of every
// query group (groups have at least two warps).
size_t probe_group_smem_bytes(uint32_t R, uint32_t S, int wpb) {
    return (size_t)((QK_CTL + R * S + 3u) & ~3u) * 4 * (wpb / 2 > 0 ? wpb / 2 : 1);
}

int probe_max_blocks_per_sm(int V, int G, uint32_t eta, int mode, int warps_per_block, size_t smem) {
    const ProbeKernel f = probe_kernel(V, G, eta, mode);
    int nb = 0;
    if (!f || (smem > 48 * 1024 &&
               cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, warps_per_block * 32, smem) != cudaSuccess)
        return 0;
    return nb;
}

cudaError_t launch_probe(const IndexView& ix, const HashParams& hp, const BatchView& b, const QueryOut& o,
                         const QueryTuning& t, DevStatus* st, cudaStream_t s, int* n_launched) {
    *n_launched = 0;
    if (b.n == 0 && !b.desc) return cudaSuccess;
    if (t.wide) {
        *n_launched = 1;
        return launch_query_wide(ix, hp, b, o, t.blocks, st, s);
    }
    // Which instances the batch needs: known here for a batch sized on the
    // host.  For one sized on the device every instance that can be the
    // batch's is launched, and the others return at once (a plan's sequences
    // are not worth the third one: they rarely have just eight k-mers).
    const int group = t.probe_blocks_group > 0 ? t.group : 1;
    bool run[3] = {true, t.probe_blocks_group > 0, !(b.desc && b.seq) && group <= 1 && b.n >= PB_MANY};
    const unsigned wpb = (unsigned)t.probe_group_wpb;
    if (b.ends && qk_group_size(b.n, group, wpb, t.probe_group_warps, 1) == 1) run[PB_GROUP] = false;
    if (!b.desc && !b.ends) {
        unsigned P;
        const int mode = probe_mode(b, group, wpb, t.probe_group_warps, 1, P);
        for (int m = 0; m < 3; ++m) run[m] = m == mode;
        // with lane groups, also for queries longer than they take, if there can be one
        const uint64_t least = b.seq ? b.k : 1;
        if (mode == PB_LANES) run[PB_WARP] = b.total > (b.n - 1) * least + (least - 1) + PB_SHORT_MOST;
    }
    for (const int mode : {PB_LANES, PB_WARP, PB_GROUP}) {
        if (!run[mode]) continue;
        const ProbeKernel f = probe_kernel(t.V, t.G, ix.eta, mode);
        if (!f) return cudaErrorInvalidValue;
        const unsigned threads = (unsigned)(mode == PB_GROUP ? t.probe_group_wpb : t.probe_warps) * 32;
        const size_t smem = mode == PB_GROUP ? probe_group_smem_bytes(ix.R, ix.S, t.probe_group_wpb) : 0;
        const int blocks = mode == PB_GROUP ? t.probe_blocks_group : mode == PB_LANES ? t.probe_blocks_lanes : t.probe_blocks;
        f<<<(unsigned)blocks, threads, smem, s>>>(ix, hp, b, o, t.probe_batch, t.order, group, t.probe_group_wpb,
                                                  t.probe_group_warps, run[PB_LANES] ? 1 : 0, st);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        ++*n_launched;
    }
    return cudaSuccess;
}

}  // namespace rgb
