// k_probe_e2.cu -- probe kernel instances for up to two hashes per filter.
#define QK_ETA 2
#define QK_SUFFIX e2
#include "k_probe_inst.cuh"
