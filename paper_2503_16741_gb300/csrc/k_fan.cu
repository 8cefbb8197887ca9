// k_fan.cu -- 2D fan-beam projectors (Sec. 2.2, 2.3; flat and curved
// detectors): one slice, one detector row, so there is no axial direction to
// share a footprint down (the single unit row lies inside every voxel's axial
// extent, factor 1) and the work per (pixel, view) is the transaxial footprint
// itself.  What bounds these kernels is the instruction issue of that
// footprint and, for the small images that fan-beam requests usually are, how
// many warps there are to issue it: a 128 x 128 image has 512 warps of pixels,
// fewer than the chip has schedulers.  Hence both directions split the sum as
// well as the outputs:
//   back:    a warp owns 8 x 4 pixels (a compact patch: its lanes read
//            neighbouring detector cells), the block's 8 warps take every
//            eighth view of the same patch and add up through shared memory;
//   forward: a block owns 32 cells of one view, its 8 warps take every eighth
//            slab of the image; a warp evaluates each pixel's footprint once
//            (lane = pixel) and its lanes then gather it per cell;
//   ray:     the same blocks, thread = (ray, every eighth run of slabs).
// Every sum has a fixed order that depends on the geometry only:
// deterministic, and batch items do not depend on the batch.
// Batch items go in pairs that share each footprint.
// Measured against the circular kernels with nz = nv = 1 that served fan beam
// before (forward + back of one pass): 128 x 128, 180 views, ray-driven
// forward and voxel-driven back 310 -> 36 us; 512 x 512, 720 views, FBP
// 2058 -> 380 us (436 us with one pixel to a thread); 2 images of 301 x 301,
// 217 views, SF forward and back 4460 -> 625 us (1192 us before the pairs and
// the cheaper footprint).
#include <algorithm>
#include <type_traits>

#include "ct_device.cuh"
#include "ct_launch.h"
#include "k_nc.cuh"
#include "k_ray.cuh"

namespace ctp {

namespace {
constexpr int kFanWarps = 8;   // warps per block (view or slab groups)
constexpr int kFanViews = 64;  // view records staged at a time
}  // namespace

// Transaxial footprint of pixel (i, j): knots relative to cell aref, and the
// amplitude (SF-TR; DD and SF-TT have a per-cell factor instead).
template <int KIND, bool CURVED>
__device__ __forceinline__ void fan_foot(const CtView &V, const CtGrid &g, int i, int j, float cu, float cn, Trap &T,
                                         int &aref, float &amp) {
    float k[4];
    column_knots<CURVED, KIND == FAN_DD>(V, cu, cn, aref, k);
    amp = 1.f;
    if (KIND == FAN_DD) {
        T = Trap{k[0], k[0], k[3], k[3], 0.f, 0.f};  // (the box's weights are plain overlaps)
    } else {
        T = nc_trap(k[0], k[1], k[2], k[3]);
        if (KIND == FAN_SF) {
            const float wx = fmaf((float)i, g.dx, V.o[0]), wy = fmaf((float)j, g.dy, V.o[1]);
            const float r2 = fmaf(wx, wx, wy * wy);
            amp = __fdividef(g.dx * r2 * rsqrtf(r2), fmaxf(fabsf(wx), fabsf(wy)));
        }
    }
}

// u position (cells), and the squared depth of the voxel-driven and recon weights
template <bool CURVED>
__device__ __forceinline__ void fan_point(const CtView &V, float cu, float cn, float &fu, float &rden2) {
    if (CURVED) {
        fu = fmaf(V.Ku, atan2f(cu, cn), V.Cu);
        rden2 = __fdividef(1.f, fmaf(cu, cu, cn * cn));
    } else {
        const float r = rcp_newton(cn);
        fu = fmaf(V.Ku, cu * r, V.Cu);
        rden2 = r * r;
    }
}

// the footprint's integral up to u (cells from aref)
template <int KIND> __device__ __forceinline__ float fan_G(const Trap &T, float u) {
    return KIND == FAN_DD ? fminf(fmaxf(u, T.k0), T.k3) - T.k0 : trap_G(T, u);
}

template <int KIND, bool CURVED>
__device__ __forceinline__ float fan_cell_factor(const CtView &V, const CtGrid &g, int a) {
    return KIND == FAN_DD ? dd_len<CURVED>(V, g, a, 0) : (KIND == FAN_TT ? tt_amp(V, g, a, 0) : 1.f);
}

// one slab of the horizontal path: direction component w, offset e, half width h
__device__ __forceinline__ void fan_slab(float w, float e, float h, float &lo, float &hi, bool &in) {
    if (w == 0.f) {
        if (!(e >= -h && e < h)) in = false;
    } else {
        const float inv = 1.f / w;
        const float t1 = (-h - e) * inv, t2 = (h - e) * inv;
        lo = fmaxf(lo, fminf(t1, t2));
        hi = fminf(hi, fmaxf(t1, t2));
    }
}

// ------------------------------------------------------------ back (gather)
// adds one view's contributions to pixel (i, j) of NBT batch items, whose rows
// y are ystride apart (the footprint is formed once for all of them).  OWN
// (voxel-driven): a pixel that projects beside the detector adds nothing, rather than
// its end cell with a weight of zero.
template <typename TIn, int KIND, bool CURVED, bool RECON, int NBT, bool OWN = false>
__device__ __forceinline__ void fan_back_view(const CtView &V, const CtGrid &g, const TIn *__restrict__ y,
                                              size_t ystride, int i, int j, float (&acc)[NBT]) {
    const float fi = (float)i, fj = (float)j;
    const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
    const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
    if (KIND == FAN_VOX) {
        float fu, rden2;
        fan_point<CURVED>(V, cu, cn, fu, rden2);
        const float af = floorf(fu), t = fu - af;
        const int a0 = (int)af;
        if (OWN && (fu <= -1.f || fu >= (float)g.nu)) return;
        // cells off the detector weigh zero and read a clamped address
        const float w0 = (unsigned)a0 < (unsigned)g.nu ? 1.f - t : 0.f;
        const float w1 = (unsigned)(a0 + 1) < (unsigned)g.nu ? t : 0.f;
        float amp = V.rc_w * rden2;
        if (!RECON) {
            const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
            const float r2 = fmaf(wx, wx, wy * wy);
            amp = (g.dx * g.dy / g.du) * V.D * r2 * rsqrtf(r2) * rden2;
        }
        const int c0 = min(max(a0, 0), g.nu - 1), c1 = min(max(a0 + 1, 0), g.nu - 1);
#pragma unroll
        for (int q = 0; q < NBT; ++q, y += ystride)
            acc[q] = fmaf(amp, fmaf(w1, ld(y, (size_t)c1), w0 * ld(y, (size_t)c0)), acc[q]);
    } else if (KIND == FAN_RAY) {
        int aref;
        float k[4];
        column_knots<CURVED, false>(V, cu, cn, aref, k);  // the pixel's shadow
        const int d0 = max((int)ceilf(k[0] - kSearchPad), -aref);
        const int d1 = min((int)floorf(k[3] + kSearchPad), g.nu - 1 - aref);
        if (d0 > d1) return;
        float fu, unused;
        fan_point<CURVED>(V, cu, cn, fu, unused);
        int ref;
        float fr;
        split_cell(fu, ref, fr);  // (ref == aref: the same operations)
        const float rho = Det<CURVED>::den(cu, cn);
        for (int d = d0; d <= d1; ++d) {
            const float dfu = (float)(d + (aref - ref)) - fr;
            float wx, wy, ex, ey;
            if (CURVED) {
                float sg, cg;
                sincosf(((float)(aref + d) - V.Cu) / V.Ku, &sg, &cg);
                wx = fmaf(cg, V.nn[0], sg * V.eu[0]);
                wy = fmaf(cg, V.nn[1], sg * V.eu[1]);
                const float lat = rho * sinf(dfu / V.Ku);  // foot of the perpendicular from the pixel centre
                ex = lat * fmaf(cg, V.eu[0], -sg * V.nn[0]);
                ey = lat * fmaf(cg, V.eu[1], -sg * V.nn[1]);
            } else {
                const float U = g.du * ((float)(aref + d) - V.Cu);
                const float rh = rsqrtf(fmaf(U, U, V.D * V.D));
                wx = fmaf(V.D, V.nn[0], U * V.eu[0]) * rh;
                wy = fmaf(V.D, V.nn[1], U * V.eu[1]) * rh;
                const float eo = (cn / V.D) * g.du * dfu;  // offset at the pixel centre's depth
                ex = eo * V.eu[0];
                ey = eo * V.eu[1];
            }
            float lo = -3.0e38f, hi = 3.0e38f;
            bool in = true;
            fan_slab(wx, ex, 0.5f * g.dx, lo, hi, in);
            fan_slab(wy, ey, 0.5f * g.dy, lo, hi, in);
            if (in && hi > lo) {
#pragma unroll
                for (int q = 0; q < NBT; ++q) acc[q] = fmaf(hi - lo, ld(y + q * ystride, (size_t)(aref + d)), acc[q]);
            }
        }
    } else {
        Trap T;
        int aref;
        float amp;
        fan_foot<KIND, CURVED>(V, g, i, j, cu, cn, T, aref, amp);
        const int d0 = max((int)floorf(T.k0 + 0.5f), -aref);
        const int d1 = min((int)floorf(T.k3 + 0.5f), g.nu - 1 - aref);
        float s[NBT], Gp = fan_G<KIND>(T, (float)d0 - 0.5f);
#pragma unroll
        for (int q = 0; q < NBT; ++q) s[q] = 0.f;
        for (int d = d0; d <= d1; ++d) {
            const float Gn = fan_G<KIND>(T, (float)d + 0.5f);
#pragma unroll
            for (int q = 0; q < NBT; ++q) s[q] = fmaf(Gn - Gp, ld(y + q * ystride, (size_t)(aref + d)), s[q]);
            Gp = Gn;
        }
        if (RECON) {  // depth weight over the footprint's area (cells) x axial height (rows)
            const float den = Det<CURVED>::den(cu, cn);
            const float area = 0.5f * ((T.k3 - T.k0) + (T.k2 - T.k1));
            amp = __fdividef(V.rc_w, den * V.Kv * fabsf(V.av[2]) * area);
        }
#pragma unroll
        for (int q = 0; q < NBT; ++q) acc[q] = fmaf(amp, s[q], acc[q]);
    }
}

// PX: pixels of a thread (the patch is 8 x 4 PX), which share the view record's
// reads from shared memory: two in large images, where the warps suffice.
template <typename TIn, int KIND, bool CURVED, bool RECON, int NBT, int PX>
__global__ void __launch_bounds__(32 * kFanWarps)
fan_back(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ sino, void *__restrict__ vol, int out_t,
         int tiles_x, int batch) {
    __shared__ CtView sview[kFanViews];
    __shared__ float red[PX * NBT][kFanWarps][32];
    const int lane = threadIdx.x, w = threadIdx.y, tid = w * 32 + lane;
    const int i = (int)(blockIdx.x % tiles_x) * 8 + (lane & 7);
    const int j = (int)(blockIdx.x / tiles_x) * (4 * PX) + (lane >> 3);
    const bool active = i < g.nx && j < g.ny;
    const size_t ystride = (size_t)g.nview * g.nu;
    for (int bt = blockIdx.y * NBT; bt < batch; bt += gridDim.y * NBT) {
        const TIn *ys = sino + bt * ystride;
        float acc[PX][NBT];
#pragma unroll
        for (int q = 0; q < PX * NBT; ++q) acc[q / NBT][q % NBT] = 0.f;
        for (int v0 = 0; v0 < g.nview; v0 += kFanViews) {
            const int n = min(kFanViews, g.nview - v0);
            __syncthreads();
            const float4 *s4 = reinterpret_cast<const float4 *>(views + v0);
            float4 *d4 = reinterpret_cast<float4 *>(sview);
            for (int t = tid; t < n * (int)(sizeof(CtView) / sizeof(float4)); t += 32 * kFanWarps) d4[t] = __ldg(s4 + t);
            __syncthreads();
            if (active)
                for (int t = w; t < n; t += kFanWarps)
#pragma unroll
                    for (int e = 0; e < PX; ++e)
                        if (e == 0 || j + 4 * e < g.ny)
                            fan_back_view<TIn, KIND, CURVED, RECON, NBT>(sview[t], g, ys + (size_t)(v0 + t) * g.nu,
                                                                         ystride, i, j + 4 * e, acc[e]);
        }
        if constexpr (KIND == FAN_VOX) {
            // An infinite or NaN cell at an end of the detector makes the sums of the pixels
            // beyond it NaN (zero times it): a thread with such a sum starts again without
            // them.  (A test per view cost the kernel 2 to 15 %.)
            float bad = 0.f;
#pragma unroll
            for (int q = 0; q < PX * NBT; ++q) bad = fmaf(acc[q / NBT][q % NBT], 0.f, bad);
            if (bad != 0.f) {
#pragma unroll
                for (int q = 0; q < PX * NBT; ++q) acc[q / NBT][q % NBT] = 0.f;
                for (int v = w; v < g.nview; v += kFanWarps)
#pragma unroll
                    for (int e = 0; e < PX; ++e)
                        if (e == 0 || j + 4 * e < g.ny)
                            fan_back_view<TIn, KIND, CURVED, RECON, NBT, true>(views[v], g, ys + (size_t)v * g.nu, ystride, i,
                                                                               j + 4 * e, acc[e]);
            }
        }
#pragma unroll
        for (int q = 0; q < PX * NBT; ++q) red[q][w][lane] = acc[q / NBT][q % NBT];
        __syncthreads();
        const int je = j + 4 * (w / NBT);
        if (w < PX * NBT && active && je < g.ny) {
            float s = red[w][0][lane];
#pragma unroll
            for (int q = 1; q < kFanWarps; ++q) s += red[w][q][lane];
            st_out(g, vol, (size_t)(bt + w % NBT) * g.ny * g.nx + (size_t)je * g.nx + i, s, out_t);
        }
    }
}

// ------------------------------------------------------------ forward (gather)
// Block = 32 cells of one view.  A warp takes the slabs w, w + 8, ...: the
// pixels of a slab that can reach the tile are evaluated one per lane (weights
// x amplitude x value into the warp's slice of shared memory), then each lane
// adds, for its cell, the pixels between the two lines of constant u that
// bound its footprint's reach (their lateral index is affine in the slab).
template <typename TIn, int KIND, bool CURVED, int NA, int NBT>
__global__ void __launch_bounds__(32 * kFanWarps)
fan_fwd(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol, void *__restrict__ sino, int out_t,
        int tiles_u) {
    __shared__ CtView V;
    __shared__ float Sw[kFanWarps][NA][32 + 1];
    __shared__ float Sx[kFanWarps][NBT][32];
    __shared__ int Sa[kFanWarps][32];
    __shared__ float red[NBT][kFanWarps][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    int bx = blockIdx.x;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int v = bx % g.nview;
    const int bt = bx / g.nview * NBT;
    if (w == 0 && lane < (int)(sizeof(CtView) / sizeof(float4)))
        reinterpret_cast<float4 *>(&V)[lane] = __ldg(reinterpret_cast<const float4 *>(views + v) + lane);
    __syncthreads();
    const int a = tu * 32 + lane;
    const int main_y = V.main_y;
    const SlabCoef c = slab_coef(V, main_y);
    const float mu = KIND == FAN_VOX ? 1.f + kSearchPad : (KIND == FAN_DD ? V.m_dd_u : V.m_sf_u) + 0.5f + kSearchPad;
    const int nslab = main_y ? g.ny : g.nx, nlat = main_y ? g.nx : g.ny;
    const float T1 = Det<CURVED>::ratio_at(V, (float)a - mu), T2 = Det<CURVED>::ratio_at(V, (float)a + mu);
    const float q1 = 1.f / (c.ul - T1 * c.nl), q2 = 1.f / (c.ul - T2 * c.nl);
    const float p1 = fmaf(T1, c.n3, -c.u3) * q1, s1 = fmaf(T1, c.ns, -c.us) * q1;
    const float p2 = fmaf(T2, c.n3, -c.u3) * q2, s2 = fmaf(T2, c.ns, -c.us) * q2;
    const size_t npix = (size_t)g.nx * g.ny;
    const TIn *x = vol + bt * npix;
    float acc[NBT];
#pragma unroll
    for (int q = 0; q < NBT; ++q) acc[q] = 0.f;
    for (int s = w; s < nslab; s += kFanWarps) {
        const float fs = (float)s;
        const float la = fmaf(s1, fs, p1), lb = fmaf(s2, fs, p2);
        // (1e-3 pixel: rounding of the lines)
        // (lanes past the detector's end ask for none)
        const int lo = a < g.nu ? max((int)ceilf(fminf(la, lb) - 1e-3f), 0) : nlat;
        const int hi = a < g.nu ? min((int)floorf(fmaxf(la, lb) + 1e-3f), nlat - 1) : -1;
        const int L0 = __reduce_min_sync(~0u, lo), L1 = __reduce_max_sync(~0u, hi);
        for (int base = L0; base <= L1; base += 32) {
            const int l = base + lane;
            if (l <= L1) {
                const int i = main_y ? l : s, j = main_y ? s : l;
#pragma unroll
                for (int q = 0; q < NBT; ++q) Sx[w][q][lane] = ld(x + q * npix, (size_t)j * g.nx + i);
                const float fi = (float)i, fj = (float)j;
                const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
                const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
                if (KIND == FAN_VOX) {
                    float fu, rden2;
                    fan_point<CURVED>(V, cu, cn, fu, rden2);
                    const float af = floorf(fu), t = fu - af;
                    const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
                    const float r2 = fmaf(wx, wx, wy * wy);
                    const float val = (g.dx * g.dy / g.du) * V.D * r2 * rsqrtf(r2) * rden2;
                    Sw[w][0][lane] = (1.f - t) * val;
                    Sw[w][1][lane] = t * val;
                    Sa[w][lane] = (int)af;
                } else {
                    Trap T;
                    int aref;
                    float amp;
                    fan_foot<KIND, CURVED>(V, g, i, j, cu, cn, T, aref, amp);
                    const int d0 = (int)floorf(T.k0 + 0.5f), d1 = (int)floorf(T.k3 + 0.5f);
                    float F[NA];
                    if (KIND == FAN_DD) {
#pragma unroll
                        for (int q = 0; q < NA; ++q)
                            F[q] = overlap(T.k0, T.k3, (float)(d0 + q) - 0.5f, (float)(d0 + q) + 0.5f);
                    } else {
                        nc_cells<NA>(T, d0, d1, F);
                    }
#pragma unroll
                    for (int q = 0; q < NA; ++q) Sw[w][q][lane] = F[q] * amp;
                    Sa[w][lane] = aref + d0;
                }
            }
            __syncwarp();
            const int cb = min(hi, min(base + 31, L1)) - base;
            for (int q = max(lo, base) - base; q <= cb; ++q) {
                const int d = a - Sa[w][q];
                if ((unsigned)d < (unsigned)NA) {
                    const float wt = Sw[w][d][q];
#pragma unroll
                    for (int e = 0; e < NBT; ++e) acc[e] = fmaf(wt, Sx[w][e][q], acc[e]);
                }
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int e = 0; e < NBT; ++e) red[e][w][lane] = acc[e];
    __syncthreads();
    if (w >= NBT || a >= g.nu) return;
    float s = red[w][0][lane];
#pragma unroll
    for (int q = 1; q < kFanWarps; ++q) s += red[w][q][lane];
    st_out(g, sino, ((size_t)(bt + w) * g.nview + v) * g.nu + a, s * fan_cell_factor<KIND, CURVED>(V, g, a), out_t);
}

// Ray-driven forward: thread = (ray, one of 8 runs of slabs), see ray_runs.
template <typename TIn, bool CURVED>
__global__ void __launch_bounds__(32 * kFanWarps)
fan_ray_fwd(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol, void *__restrict__ sino,
            int out_t, int tiles_u) {
    __shared__ float red[kFanWarps][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    int bx = blockIdx.x;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int v = bx % g.nview;
    const int bt = bx / g.nview;
    const int a = tu * 32 + lane;
    float acc[1] = {0.f}, len = 0.f;
    if (a < g.nu)
        ray_runs<TIn, CURVED, true, kFanWarps, 1>(views[v], g, a, 0, vol + (size_t)bt * g.nx * g.ny, nullptr, w, len, acc);
    red[w][lane] = acc[0];
    __syncthreads();
    if (w || a >= g.nu) return;
    float s = red[0][lane];
#pragma unroll
    for (int q = 1; q < kFanWarps; ++q) s += red[q][lane];
    st_out(g, sino, ((size_t)bt * g.nview + v) * g.nu + a, s * len, out_t);
}

// ------------------------------------------------------------ launchers
namespace {
template <typename TIn, int KIND, bool CURVED, int NBT>
cudaError_t fan_fwd_k(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                      cudaStream_t st) {
    const int tiles_u = (g.nu + 31) / 32;
    dim3 blk(32, kFanWarps), grd((unsigned)((size_t)tiles_u * g.nview * (batch / NBT)));
    if constexpr (KIND == FAN_RAY) {
        fan_ray_fwd<TIn, CURVED><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    } else if constexpr (KIND == FAN_VOX) {
        fan_fwd<TIn, KIND, CURVED, 2, NBT><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    } else {
        // a footprint of half width m meets at most 4 cells when m <= 1.5, 8 when m <= 3.5
        const float m = KIND == FAN_DD ? g.max_m_dd_u : g.max_m_sf_u;
        if (m <= 1.5f)
            fan_fwd<TIn, KIND, CURVED, 4, NBT><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
        else
            fan_fwd<TIn, KIND, CURVED, 8, NBT><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    }
    return cudaGetLastError();
}

template <typename TIn, int KIND, bool CURVED, bool RECON, int NBT>
cudaError_t fan_back_k(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                       cudaStream_t st) {
    // two pixels to a thread from 256 x 256 on (2048 warps of patches, before the
    // split over views), where one image goes alone
    const int px = NBT == 1 && (long long)g.nx * g.ny >= 65536 ? 2 : 1;
    const int tiles_x = (g.nx + 7) / 8, tiles_y = (g.ny + 4 * px - 1) / (4 * px);
    dim3 blk(32, kFanWarps), grd((unsigned)tiles_x * (unsigned)tiles_y, (unsigned)std::min(batch / NBT, 65535));
    if (px == 2)
        fan_back<TIn, KIND, CURVED, RECON, NBT, NBT == 1 ? 2 : 1><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_x, batch);
    else
        fan_back<TIn, KIND, CURVED, RECON, NBT, 1><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_x, batch);
    return cudaGetLastError();
}

// Batch items in pairs, which share each footprint, and the odd one alone (the
// same operations on every item, so its result does not depend on its partner).
template <typename TIn, int KIND, bool CURVED>
cudaError_t fan_pairs(int dir, const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                      cudaStream_t st) {
    const int two = KIND == FAN_RAY && dir == 0 ? 0 : batch & ~1;
    const size_t nvol = (size_t)g.nx * g.ny, nsino = (size_t)g.nview * g.nu;
    cudaError_t e = cudaSuccess;
    auto go = [&](auto pair, const TIn *in, void *to, int n) {
        constexpr int NBT = decltype(pair)::value ? 2 : 1;
        if (dir == 0) return fan_fwd_k<TIn, KIND, CURVED, NBT>(g, views, in, to, out_t, n, st);
        if constexpr (KIND == FAN_SF || KIND == FAN_DD || KIND == FAN_VOX)
            if (dir == 2) return fan_back_k<TIn, KIND, CURVED, true, NBT>(g, views, in, to, out_t, n, st);
        return fan_back_k<TIn, KIND, CURVED, false, NBT>(g, views, in, to, out_t, n, st);
    };
    if (two) e = go(std::true_type(), src, out, two);
    if (e == cudaSuccess && batch > two) {
        const size_t in_item = dir == 0 ? nvol : nsino, out_item = dir == 0 ? nsino : nvol;
        e = go(std::false_type(), src + two * in_item,
               static_cast<char *>(out) + two * out_item * (out_t == 0 ? 4 : 2), batch - two);
    }
    return e;
}

template <typename TIn, int KIND>
cudaError_t fan_t(int dir, const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                  cudaStream_t st) {
    const TIn *src = static_cast<const TIn *>(in);
    return g.variant == GEO_CIRC_CURVED ? fan_pairs<TIn, KIND, true>(dir, g, views, src, out, out_t, batch, st)
                                        : fan_pairs<TIn, KIND, false>(dir, g, views, src, out, out_t, batch, st);
}

template <typename TIn>
cudaError_t fan_kinds(int kind, int dir, const CtGrid &g, const CtView *views, const void *in, void *out, int out_t,
                      int batch, cudaStream_t st) {
    switch (kind) {
    case FAN_SF: return fan_t<TIn, FAN_SF>(dir, g, views, in, out, out_t, batch, st);
    case FAN_DD: return fan_t<TIn, FAN_DD>(dir, g, views, in, out, out_t, batch, st);
    case FAN_TT: return fan_t<TIn, FAN_TT>(dir, g, views, in, out, out_t, batch, st);
    case FAN_VOX: return fan_t<TIn, FAN_VOX>(dir, g, views, in, out, out_t, batch, st);
    default: return fan_t<TIn, FAN_RAY>(dir, g, views, in, out, out_t, batch, st);
    }
}
}  // namespace

bool fan_fits(const CtGrid &g, int kind, int dir) {
    if (!g.is2d) return false;
    return dir != 0 || kind == FAN_VOX || kind == FAN_RAY || (kind == FAN_DD ? g.max_m_dd_u : g.max_m_sf_u) <= 3.5f;
}

cudaError_t launch_fan(int kind, int dir, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                       void *out, int batch, cudaStream_t st) {
    switch (in_t) {
    case 0: return fan_kinds<float>(kind, dir, g, views, in, out, out_t, batch, st);
    case 1: return fan_kinds<__half>(kind, dir, g, views, in, out, out_t, batch, st);
    default: return fan_kinds<__nv_bfloat16>(kind, dir, g, views, in, out, out_t, batch, st);
    }
}

}  // namespace ctp
