// k_circ_fwd_f32.cu -- the circular forward projection (k_circ_fwd.cuh) of F32
// volumes and its launcher; one storage type per translation unit, compiled in parallel.
#include "k_circ_fwd.cuh"

namespace ctp {

// a[k/4][j][i][k%4] = b[k/4][i][j][k%4] = x[k][j][i], zero from nz on (either may be
// null): CTA = 32 x 32 columns of one group of four slices, both copies from one read
template <typename T>
__global__ void __launch_bounds__(256)
quad_copies(const T *__restrict__ x, T *__restrict__ ya, T *__restrict__ xb, int nx, int ny, int nz, int nzp) {
    struct alignas(4 * sizeof(T)) Quad { T v[4]; };
    __shared__ Quad tile[32][33];
    const int tiles_i = (nx + 31) / 32;
    const int i0 = (blockIdx.x % tiles_i) * 32, j0 = (blockIdx.x / tiles_i) * 32, k0 = blockIdx.y * 4;
    const size_t ncol = (size_t)nx * ny;
    const T *src = x + (size_t)blockIdx.z * ncol * nz;
    const size_t at = ((size_t)blockIdx.z * (nzp / 4) + blockIdx.y) * ncol;
    Quad *a = ya ? reinterpret_cast<Quad *>(ya) + at : nullptr, *b = xb ? reinterpret_cast<Quad *>(xb) + at : nullptr;
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = i0 + threadIdx.x, j = j0 + r;
        if (i >= nx || j >= ny) continue;
        Quad q;
#pragma unroll
        for (int t = 0; t < 4; ++t) q.v[t] = k0 + t < nz ? src[(size_t)(k0 + t) * ncol + (size_t)j * nx + i] : T(0.f);
        if (a) a[(size_t)j * nx + i] = q;
        tile[r][threadIdx.x] = q;
    }
    if (!b) return;  // (uniform)
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += 8) {
        const int i = i0 + r, j = j0 + threadIdx.x;
        if (i < nx && j < ny) b[(size_t)i * ny + j] = tile[threadIdx.x][r];
    }
}

cudaError_t circ_fwd_f16(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t,
                         int batch, cudaStream_t st);
cudaError_t circ_fwd_bf16(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out,
                          int out_t, int batch, cudaStream_t st);

cudaError_t circ_fwd_f32(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t,
                         int batch, cudaStream_t st) {
    return circ_fwd_kind<float>(kind, g, views, x, out, out_t, batch, st);
}

// (voxels of 64 rows and more would spend their time on whole rows)
bool circ_fwd_fits(const CtGrid &g, int kind, int batch) {
    if (zmajor_pitch(g) == 0 || batch > 65535 || !(g.max_m_sf_v < 32.f)) return false;
    return kind == BK_VOX || (kind == BK_DD ? g.max_m_dd_u : g.max_m_sf_u) <= 3.5f;
}

namespace {
size_t copy_bytes(const CtGrid &g, int batch, int elem_bytes) {
    return (size_t)g.nx * g.ny * zmajor_pitch(g) * batch * elem_bytes;
}
template <typename T>
cudaError_t make_copies(const CtGrid &g, const void *x, void *a, void *b, int batch, cudaStream_t st) {
    const int nzp = zmajor_pitch(g);
    const dim3 tg((unsigned)(((g.nx + 31) / 32) * ((g.ny + 31) / 32)), (unsigned)(nzp / 4), (unsigned)batch);
    quad_copies<T><<<tg, dim3(32, 8), 0, st>>>(static_cast<const T *>(x), static_cast<T *>(a), static_cast<T *>(b), g.nx, g.ny,
                                               g.nz, nzp);
    return cudaGetLastError();
}
}  // namespace

// A copy for each main axis that the views have; with memory for one of two, each in
// turn in the same buffer, before a launch of its views (256^3 / 360 views SF-TR 11.1
// against 10.6 ms); with memory for none, the volume in place (27 ms).  The
// results are the same.
size_t circ_fwd_workspace(const CtGrid &g, int batch, int elem_bytes) {
    if (circ_fwd_direct(g, batch)) return 0;
    return copy_bytes(g, batch, elem_bytes) * (g.axes == 3 ? 2 : 1);
}

cudaError_t launch_circ_fwd(int kind, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                            void *out, int batch, cudaStream_t st) {
    const int isz = in_t == 0 ? 4 : 2;
    auto go = [&](const FwdVolume &x) {
        switch (in_t) {
        case 0: return circ_fwd_f32(kind, g, views, x, out, out_t, batch, st);
        case 1: return circ_fwd_f16(kind, g, views, x, out, out_t, batch, st);
        default: return circ_fwd_bf16(kind, g, views, x, out, out_t, batch, st);
        }
    };
    auto copy = [&](void *a, void *b) {  // (bit patterns of either half type; the padding is zero in both)
        return in_t == 0 ? make_copies<float>(g, in, a, b, batch, st) : make_copies<__half>(g, in, a, b, batch, st);
    };
    const size_t one = copy_bytes(g, batch, isz);
    char *buf = nullptr;
    int copies = circ_fwd_direct(g, batch) ? 0 : g.axes == 3 ? 2 : 1;
    for (; copies > 0; --copies) {
        if (workspace_alloc_copy((void **)&buf, one * copies, g, st) == cudaSuccess) break;
        cudaGetLastError();
        buf = nullptr;
    }
    if (copies == 0) return go(FwdVolume{in, in, 0});
    const int nzp = zmajor_pitch(g);
    cudaError_t e = cudaSuccess;
    if (copies == 2 || g.axes != 3) {
        char *y = g.axes & 1 ? buf : nullptr, *x = g.axes & 2 ? buf + (copies - 1) * one : nullptr;
        e = copy(y, x);
        if (e == cudaSuccess) e = go(FwdVolume{y, x, nzp});
    } else {
        e = copy(buf, nullptr);
        if (e == cudaSuccess) e = go(FwdVolume{buf, nullptr, nzp});
        if (e == cudaSuccess) e = copy(nullptr, buf);
        if (e == cudaSuccess) e = go(FwdVolume{nullptr, buf, nzp});
    }
    const cudaError_t ef = workspace_free(buf, st);
    return e != cudaSuccess ? e : ef;
}

}  // namespace ctp
