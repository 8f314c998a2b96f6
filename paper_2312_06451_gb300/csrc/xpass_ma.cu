// Pass kernels: multi-angle.
#include "xpass.cuh"

namespace qg {

cudaError_t launch_xpass_ma(int bwd, int cost_dtype, int nbuf, int gather, const PassDesc *d, const uint32_t *tb,
                 int nd, uint32_t tiles, int *err, uint32_t *sched, cudaStream_t s) {
    return launch_xpass_g<1, 0>(bwd, cost_dtype, nbuf, gather, d, tb, nd, tiles, err, sched, s);
}

}  // namespace qg
