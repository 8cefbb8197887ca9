// k_circ_back_f16.cu -- the circular backprojection (k_circ_back.cuh) of F16
// sinograms; one storage type per translation unit, compiled in parallel.
#include "k_circ_back.cuh"

namespace ctp {

cudaError_t circ_back_f16(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                          int out_t, int batch, cudaStream_t st) {
    return circ_back_kind<__half>(kind, recon, g, views, in, out, out_t, batch, st);
}

}  // namespace ctp
