// k_circ_back_f32.cu -- the circular backprojection (k_circ_back.cuh) of F32
// sinograms and its dispatch; one storage type per translation unit, compiled in parallel.
#include "k_circ_back.cuh"

namespace ctp {

cudaError_t circ_back_f16(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                          int out_t, int batch, cudaStream_t st);
cudaError_t circ_back_bf16(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                           int out_t, int batch, cudaStream_t st);

cudaError_t circ_back_f32(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                          int out_t, int batch, cudaStream_t st) {
    return circ_back_kind<float>(kind, recon, g, views, in, out, out_t, batch, st);
}

// nu >= 8: a window of 8 cells fits the detector
bool circ_back_fits(const CtGrid &g, int kind) {
    if (g.is2d || g.variant == GEO_NONCIRC_FLAT || g.nu < 8 || !(g.max_m_sf_v < 4.f)) return false;
    return kind == BK_VOX || (kind == BK_DD ? g.max_m_dd_u : g.max_m_sf_u) <= 3.5f;
}

cudaError_t launch_circ_back(int kind, bool recon, const CtGrid &g, const CtView *views, int in_t, const void *in,
                             int out_t, void *out, int batch, cudaStream_t st) {
    switch (in_t) {
    case 0: return circ_back_f32(kind, recon, g, views, in, out, out_t, batch, st);
    case 1: return circ_back_f16(kind, recon, g, views, in, out, out_t, batch, st);
    default: return circ_back_bf16(kind, recon, g, views, in, out, out_t, batch, st);
    }
}

}  // namespace ctp
