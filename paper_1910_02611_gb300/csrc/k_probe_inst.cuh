// k_probe_inst.cuh -- instantiates k_probe<V, G, ETA> for one ETA (the
// including file defines QK_ETA and QK_SUFFIX), for the tilings of
// k_query_inst.cuh's list.
#pragma once
#include "k_probe.cuh"

#define QK_VG_LIST(X) \
    X(1, 1) X(2, 1) X(1, 2) X(4, 1) X(2, 2) X(4, 2) X(2, 4) X(4, 4) X(2, 8) X(1, 16) X(4, 8) X(4, 16) X(4, 32)

#define QK_CAT2(a, b) a##b
#define QK_CAT(a, b) QK_CAT2(a, b)

namespace rgb {

using ProbeKernel = void (*)(IndexView, HashParams, BatchView, QueryOut, int, int, int, int, unsigned long long, int,
                             DevStatus*);

ProbeKernel QK_CAT(probe_kernel_, QK_SUFFIX)(int V, int G, int mode) {
#define X(v, g)                                                                     \
    if (V == v && G == g)                                                           \
        return mode == PB_LANES   ? &k_probe<v, g, QK_ETA, PB_LANES>                \
               : mode == PB_GROUP ? &k_probe<v, g, QK_ETA, PB_GROUP>                \
                                  : &k_probe<v, g, QK_ETA, PB_WARP>;
    QK_VG_LIST(X)
#undef X
    return nullptr;
}

}  // namespace rgb
