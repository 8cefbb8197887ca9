// k_circ_fwd_bf16.cu -- the circular forward projection (k_circ_fwd.cuh) of BF16
// volumes; one storage type per translation unit, compiled in parallel.
#include "k_circ_fwd.cuh"

namespace ctp {

cudaError_t circ_fwd_bf16(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t,
                         int batch, cudaStream_t st) {
    return circ_fwd_kind<__nv_bfloat16>(kind, g, views, x, out, out_t, batch, st);
}

}  // namespace ctp
