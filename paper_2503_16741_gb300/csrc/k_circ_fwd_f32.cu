// k_circ_fwd_f32.cu -- the circular forward projection (k_circ_fwd.cuh) of F32
// volumes and its launcher; one storage type per translation unit, compiled in parallel.
#include "k_circ_fwd.cuh"

namespace ctp {

// dst[0][k/4][j][i][k%4] = dst[1][k/4][i][j][k%4] = x[k][j][i], zero from nz on:
// CTA = 32 x 32 columns of one group of four slices, both copies from one read
template <typename T>
__global__ void __launch_bounds__(256)
quad_copies(const T *__restrict__ x, T *__restrict__ dst, int nx, int ny, int nz, int nzp) {
    struct alignas(4 * sizeof(T)) Quad { T v[4]; };
    __shared__ Quad tile[32][33];
    const int tiles_i = (nx + 31) / 32;
    const int i0 = (blockIdx.x % tiles_i) * 32, j0 = (blockIdx.x / tiles_i) * 32, k0 = blockIdx.y * 4;
    const size_t ncol = (size_t)nx * ny;
    const T *src = x + (size_t)blockIdx.z * ncol * nz;
    Quad *a = reinterpret_cast<Quad *>(dst) + ((size_t)blockIdx.z * 2 * nzp / 4 + blockIdx.y) * ncol;
    Quad *b = a + (size_t)nzp / 4 * ncol;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = i0 + threadIdx.x, j = j0 + r;
        if (i >= nx || j >= ny) continue;
        Quad q;
#pragma unroll
        for (int t = 0; t < 4; ++t) q.v[t] = k0 + t < nz ? src[(size_t)(k0 + t) * ncol + (size_t)j * nx + i] : T(0.f);
        a[(size_t)j * nx + i] = q;
        tile[r][threadIdx.x] = q;
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = i0 + r, j = j0 + threadIdx.x;
        if (i < nx && j < ny) b[(size_t)i * ny + j] = tile[threadIdx.x][r];
    }
}

cudaError_t circ_fwd_f16(int kind, const CtGrid &g, const CtView *views, const void *xZ, int nzp, void *out, int out_t,
                         int batch, cudaStream_t st);
cudaError_t circ_fwd_bf16(int kind, const CtGrid &g, const CtView *views, const void *xZ, int nzp, void *out,
                          int out_t, int batch, cudaStream_t st);

cudaError_t circ_fwd_f32(int kind, const CtGrid &g, const CtView *views, const void *xZ, int nzp, void *out, int out_t,
                         int batch, cudaStream_t st) {
    return circ_fwd_kind<float>(kind, g, views, xZ, nzp, out, out_t, batch, st);
}

// (voxels of 64 rows and more would spend their time on whole rows)
bool circ_fwd_fits(const CtGrid &g, int kind, int batch) {
    if (zmajor_pitch(g) == 0 || batch > 65535 || !(g.max_m_sf_v < 32.f)) return false;
    return kind == BK_VOX || (kind == BK_DD ? g.max_m_dd_u : g.max_m_sf_u) <= 3.5f;
}

size_t circ_fwd_workspace(const CtGrid &g, int batch, int elem_bytes) {
    if (circ_fwd_direct(g, batch)) return 0;
    return (size_t)2 * g.nx * g.ny * zmajor_pitch(g) * batch * elem_bytes;
}

cudaError_t launch_circ_fwd(int kind, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st) {
    const int nzp = zmajor_pitch(g), isz = in_t == 0 ? 4 : 2;
    auto go = [&](const void *x) {
        switch (in_t) {
        case 0: return circ_fwd_f32(kind, g, views, x, nzp, out, out_t, batch, st);
        case 1: return circ_fwd_f16(kind, g, views, x, nzp, out, out_t, batch, st);
        default: return circ_fwd_bf16(kind, g, views, x, nzp, out, out_t, batch, st);
        }
    };
    if (circ_fwd_direct(g, batch)) return go(in);
    void *xZ = nullptr;
    cudaError_t e = workspace_alloc(&xZ, circ_fwd_workspace(g, batch, isz), st);
    if (e != cudaSuccess) return e;
    const dim3 tg((unsigned)(((g.nx + 31) / 32) * ((g.ny + 31) / 32)), (unsigned)(nzp / 4), (unsigned)batch);
    if (in_t == 0)
        quad_copies<float><<<tg, dim3(32, 8), 0, st>>>(static_cast<const float *>(in), static_cast<float *>(xZ), g.nx,
                                                       g.ny, g.nz, nzp);
    else  // (bit patterns of either half type; the padding is zero in both)
        quad_copies<__half><<<tg, dim3(32, 8), 0, st>>>(static_cast<const __half *>(in), static_cast<__half *>(xZ),
                                                        g.nx, g.ny, g.nz, nzp);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = go(xZ);
    const cudaError_t ef = workspace_free(xZ, st);
    return e != cudaSuccess ? e : ef;
}

}  // namespace ctp
