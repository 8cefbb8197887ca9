// k_circ_fwd_f16.cu -- the circular forward projection (k_circ_fwd.cuh) of F16
// volumes; one storage type per translation unit, compiled in parallel.
#include "k_circ_fwd.cuh"

namespace ctp {

cudaError_t circ_fwd_f16(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t,
                         int batch, cudaStream_t st) {
    return circ_fwd_kind<__half>(kind, g, views, x, out, out_t, batch, st);
}

}  // namespace ctp
