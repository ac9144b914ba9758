// k_probe_e4.cu -- probe kernel instances for three or four hashes per filter.
#define QK_ETA 4
#define QK_SUFFIX e4
#include "k_probe_inst.cuh"
