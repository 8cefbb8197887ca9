// k_circ_back_bf16.cu -- the circular backprojection (k_circ_back.cuh) of BF16
// sinograms; one storage type per translation unit, compiled in parallel.
#include "k_circ_back.cuh"

namespace ctp {

cudaError_t circ_back_bf16(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                          int out_t, int batch, cudaStream_t st) {
    return circ_back_kind<__nv_bfloat16>(kind, recon, g, views, in, out, out_t, batch, st);
}

}  // namespace ctp
