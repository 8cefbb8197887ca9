// k_nc_back.cu -- backprojection of the non-circular SF-TR and DD footprint
// projectors and of SF-TT, and the entries for both directions (the
// footprint and the dispatch are in k_nc.cuh).
#include <cooperative_groups.h>

#include "k_nc.cuh"

namespace ctp {

// ------------------------------------------------------------ back (gather)
constexpr int kNcViews = 8;  // views staged per round

// rows b0 .. b0 + NB - 1 under the first NC of the footprint's weights
template <typename TIn, int NC, int NA, int NB>
__device__ __forceinline__ float nc_taps(const NcFp<NA, NB> &P, const TIn *__restrict__ yv, const CtGrid &g) {
    float s = 0.f;
    if (P.b0 >= 0 && P.b0 + NB <= g.nv) {  // all rows on the detector: no test per row
        const TIn *row = yv + (size_t)P.b0 * g.nu + P.a0;
#pragma unroll
        for (int q = 0; q < NB; ++q, row += g.nu)
            if (P.Fv[q] != 0.f) {
                float rs = P.Fu[0] * ld(row, 0);
#pragma unroll
                for (int c = 1; c < NC; ++c) rs = fmaf(P.Fu[c], c < P.n ? ld(row, (size_t)c) : 0.f, rs);
                s = fmaf(P.Fv[q], rs, s);
            }
        return s;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const int b = P.b0 + q;
        if (P.Fv[q] != 0.f && b >= 0 && b < g.nv) {
            const TIn *row = yv + (size_t)b * g.nu + P.a0;
            float rs = P.Fu[0] * ld(row, 0);
#pragma unroll
            for (int c = 1; c < NC; ++c) rs = fmaf(P.Fu[c], c < P.n ? ld(row, (size_t)c) : 0.f, rs);
            s = fmaf(P.Fv[q], rs, s);
        }
    }
    return s;
}

// Thread = voxel column (i, j) over ZT voxels; per view it forms what the
// column shares and runs over its voxels one at a time (the per-voxel body
// appears once in the code, which keeps the kernel within the instruction
// cache) with the voxels' sums in shared memory.  Bound by instruction
// issue.  192^3 / 250 views FP16 SF-TR 19.8 -> 15.6 ms from forming
// corner pairs with one division each and the column's share once per view;
// 64^3 / 90 views DD 637 -> 240 us, the views split over a cluster besides.
// RECON: the recon-mode (FBP) backprojection with the normalised footprint
// as the interpolation: weight rc_w / depth^2 over the footprint's area x
// height (SF-TR and DD).
template <typename TIn, int KIND, int NA, int NB, int ZT, bool RECON = false>
__global__ void __launch_bounds__(128, 8)
nc_back(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ sino, void *__restrict__ vol,
        int out_t, int tiles_x, int nzc, int S) {
    __shared__ CtView sview[kNcViews];
    __shared__ float acc[ZT][128];
    int bx = blockIdx.x;
    const int rank = bx % S; bx /= S;  // cluster rank: the block's share of the rounds of views
    const int tx = bx % tiles_x; bx /= tiles_x;
    const int kc = bx % nzc;
    const int bt = bx / nzc;
    const int i = tx * 32 + threadIdx.x;
    const int j = blockIdx.y * 4 + threadIdx.y;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const bool active = i < g.nx && j < g.ny;
    const int kbeg = kc * ZT, kend = min(kbeg + ZT, g.nz);
#pragma unroll
    for (int q = 0; q < ZT; ++q) acc[q][tid] = 0.f;
    const size_t vstride = (size_t)g.nv * g.nu;
    const TIn *ys = sino + (size_t)bt * g.nview * vstride;
    for (int v0 = rank * kNcViews; v0 < g.nview; v0 += S * kNcViews) {
        const int nvc = min(kNcViews, g.nview - v0);
        __syncthreads();
        {
            const float4 *s4 = reinterpret_cast<const float4 *>(views + v0);
            float4 *d4 = reinterpret_cast<float4 *>(sview);
            constexpr int W = sizeof(CtView) / sizeof(float4);
            for (int t = tid; t < nvc * W; t += 128) d4[t] = __ldg(s4 + t);
        }
        __syncthreads();
        if (!active) continue;
        for (int vv = 0; vv < nvc; ++vv) {
            const CtView &V = sview[vv];
            const TIn *yv = ys + (size_t)(v0 + vv) * vstride;
            const NcCol C = nc_col<KIND>(V, g, i, j);
#pragma unroll 1
            for (int k = kbeg; k < kend; ++k) {
                NcFp<NA, NB> P;
                nc_fp<KIND, NA, NB>(V, g, C, (float)k, P);
                float s = 0.f;
                if (P.a0 >= 0 && P.a0 + NA <= g.nu) {
                    // the whole window on the detector: one row pointer and
                    // predicated loads of the footprint's cells (no branches);
                    // the bound NA holds near the source, and most footprints
                    // end by their fourth cell
                    if (NA <= 4 || P.n <= 4)
                        s = nc_taps<TIn, NA < 4 ? NA : 4, NA, NB>(P, yv, g);
                    else
                        s = nc_taps<TIn, NA, NA, NB>(P, yv, g);
                } else {
                    // cells off the detector get weight 0 and a clamped
                    // (in-bounds) address; cells past the footprint are not read
                    int ac[NA];
                    float wu[NA];
#pragma unroll
                    for (int c = 0; c < NA; ++c) {
                        const int ca = P.a0 + c;
                        const bool in = ca >= 0 && ca < g.nu;
                        ac[c] = in ? ca : 0;
                        wu[c] = in ? P.Fu[c] : 0.f;
                    }
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        const int b = P.b0 + q;
                        if (P.Fv[q] != 0.f && b >= 0 && b < g.nv) {
                            const TIn *row = yv + (size_t)b * g.nu;
                            float rs = wu[0] * ld(row, (size_t)ac[0]);
#pragma unroll
                            for (int c = 1; c < NA; ++c) {
                                if (c >= P.n) break;
                                rs = fmaf(wu[c], ld(row, (size_t)ac[c]), rs);
                            }
                            s = fmaf(P.Fv[q], rs, s);
                        }
                    }
                }
                float &a = acc[k - kbeg][tid];
                a = fmaf(RECON ? V.rc_w / (P.cn * P.cn * P.size) : P.amp, s, a);
            }
        }
    }
    const size_t zs = (size_t)g.ny * g.nx;
    const size_t base = ((size_t)bt * g.nz + kbeg) * zs + (size_t)j * g.nx + i;
    if (S == 1) {
        if (!active) return;
        for (int kk = 0; kk < kend - kbeg; ++kk) st_out(g, vol, base + kk * zs, acc[kk][tid], out_t);
        return;
    }
    // the cluster's sums, in rank order: rank r stores the voxels r, r + S, ...
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    if (active)
        for (int kk = rank; kk < kend - kbeg; kk += S) {
            float s = 0.f;
            for (int r = 0; r < S; ++r) s += cl.map_shared_rank(&acc[0][0], r)[kk * 128 + tid];
            st_out(g, vol, base + kk * zs, s, out_t);
        }
    cl.sync();  // (a block's shared memory stays until all have read it)
}

namespace {
// Small volumes split the views over the blocks of a cluster (see view_split).
template <typename TIn, int KIND, int NA, int NB, bool RECON>
cudaError_t nc_back_go(const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                       cudaStream_t st) {
    constexpr int ZT = 8;
    const int tiles_x = (g.nx + 31) / 32, nzc = (g.nz + ZT - 1) / ZT, tiles_y = (g.ny + 3) / 4;
    const int S = view_split((long long)tiles_x * tiles_y * nzc * 4, (g.nview + kNcViews - 1) / kNcViews);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((size_t)S * tiles_x * nzc * batch), (unsigned)tiles_y);
    cfg.blockDim = dim3(32, 4);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = S > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, nc_back<TIn, KIND, NA, NB, ZT, RECON>, g, views, static_cast<const TIn *>(in), out,
                              out_t, tiles_x, nzc, S);
}

template <typename TIn, int KIND, int NA, int NB> struct NcBack {
    static cudaError_t go(const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                          cudaStream_t st) {
        return nc_back_go<TIn, KIND, NA, NB, false>(g, views, in, out, out_t, batch, st);
    }
};
}  // namespace

template <typename TIn, int KIND, int NA, int NB> struct NcBackRecon {
    static cudaError_t go(const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                          cudaStream_t st) {
        return nc_back_go<TIn, KIND, NA, NB, true>(g, views, in, out, out_t, batch, st);
    }
};

cudaError_t launch_nc_recon(int dd, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st) {
    const int kind = dd ? NC_DD : NC_SF;
    if (!nc_footprint_fits(g, kind)) return cudaErrorNotSupported;
    return nc_dispatch<NcBackRecon>(kind, in_t, g, views, in, out, out_t, batch, st);
}

cudaError_t launch_nc_back(int kind, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                           void *out, int batch, cudaStream_t st) {
    return nc_dispatch<NcBack>(kind, in_t, g, views, in, out, out_t, batch, st);
}

bool nc_footprint_fits(const CtGrid &g, int kind) {
    // at most 8 cells (half width <= 3.5) by 4 rows (half height <= 1.5)
    return (kind == NC_DD ? g.max_m_dd_u : g.max_m_sf_u) <= 3.5f &&
           (kind == NC_TT ? g.max_m_tt_v : g.max_m_sf_v) <= 1.5f;
}

cudaError_t launch_nc(int kind, int dir, const CtGrid &g, const CtView *views, int in_t, const void *in,
                      int out_t, void *out, int batch, cudaStream_t st) {
    return dir == 0 ? launch_nc_fwd(kind, g, views, in_t, in, out_t, out, batch, st)
                    : launch_nc_back(kind, g, views, in_t, in, out_t, out, batch, st);
}

// SF-TT: the back direction scales the sinogram by each cell's amplitude into
// a stream-ordered FP32 workspace first.  Circular flat 3D geometry takes the
// column-walk kernels of k_sf.cu (the transaxial footprint is reused down
// each column), every other flat geometry the per-voxel footprint kernels.
template <typename TIn>
__global__ void __launch_bounds__(256)
tt_prescale(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ y, float *__restrict__ yp,
            int batch) {
    const size_t nview_cells = (size_t)g.nv * g.nu;
    const size_t total = nview_cells * g.nview * batch;
    for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int a = (int)(t % g.nu);
        const int b = (int)((t / g.nu) % g.nv);
        const int v = (int)((t / nview_cells) % g.nview);
        yp[t] = tt_amp(views[v], g, a, b) * ld(y, t);
    }
}

cudaError_t launch_sftt(int dir, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                        void *out, int batch, cudaStream_t st) {
    const bool circ = sftt_circ_fits(g);
    if (dir == 0 && fan_fits(g, FAN_TT, 0)) return launch_fan(FAN_TT, 0, g, views, in_t, in, out_t, out, batch, st);
    if (dir == 0)
        return circ ? launch_sftt_circ(0, g, views, in_t, in, out_t, out, batch, st)
                    : launch_nc(NC_TT, 0, g, views, in_t, in, out_t, out, batch, st);
    const size_t n = (size_t)g.nview * g.nv * g.nu * batch;
    float *yp = nullptr;
    cudaError_t e = workspace_alloc((void **)&yp, n * sizeof(float), st);
    if (e != cudaSuccess) return e;
    const size_t want = (n + 255) / 256;
    const unsigned blocks = (unsigned)(want < 152u * 64u ? want : 152u * 64u);
    switch (in_t) {
    case 0: tt_prescale<float><<<blocks, 256, 0, st>>>(g, views, static_cast<const float *>(in), yp, batch); break;
    case 1: tt_prescale<__half><<<blocks, 256, 0, st>>>(g, views, static_cast<const __half *>(in), yp, batch); break;
    default:
        tt_prescale<__nv_bfloat16><<<blocks, 256, 0, st>>>(g, views, static_cast<const __nv_bfloat16 *>(in), yp,
                                                           batch);
        break;
    }
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = g.is2d ? launch_fan(FAN_TT, 1, g, views, 0, yp, out_t, out, batch, st)
            : circ ? launch_sftt_circ(1, g, views, 0, yp, out_t, out, batch, st)
                   : launch_nc(NC_TT, 1, g, views, 0, yp, out_t, out, batch, st);
    const cudaError_t ef = workspace_free(yp, st);
    return e != cudaSuccess ? e : ef;
}

}  // namespace ctp
