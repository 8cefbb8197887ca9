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
// Measured against the circular kernels with nz = nv = 1 that served fan beam
// before (forward + back of one pass): 128 x 128, 180 views, ray-driven
// forward and voxel-driven back 310 -> 35 us; 512 x 512, 720 views, FBP
// 2058 -> 514 us; 2 images of 301 x 301, 217 views, SF forward and back
// 4460 -> 1192 us.
#include <algorithm>

#include "ct_device.cuh"
#include "ct_launch.h"

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
    float fr;
    split_cell(Det<CURVED>::fu(V, cu, cn), aref, fr);
    if (KIND == FAN_DD) {  // boundary points +- half a pixel along the non-main axis
        const int q = V.main_y ? 0 : 1;
        const float hu = 0.5f * V.au[q], hn = 0.5f * V.an[q];
        const float e1 = fr + Det<CURVED>::dfu(V, cu, cn, -hu, -hn);
        const float e2 = fr + Det<CURVED>::dfu(V, cu, cn, hu, hn);
        T.k0 = T.k1 = fminf(e1, e2);
        T.k2 = T.k3 = fmaxf(e1, e2);
        T.h1 = T.h3 = 0.f;  // (unused: the box's weights are plain overlaps)
        amp = 1.f;
    } else {
        float t0 = fr + Det<CURVED>::dfu(V, cu, cn, V.cdu[0], V.cdn[0]);
        float t1 = fr + Det<CURVED>::dfu(V, cu, cn, V.cdu[1], V.cdn[1]);
        float t2 = fr + Det<CURVED>::dfu(V, cu, cn, V.cdu[2], V.cdn[2]);
        float t3 = fr + Det<CURVED>::dfu(V, cu, cn, V.cdu[3], V.cdn[3]);
        sort4(t0, t1, t2, t3);
        T = make_trap(t0, t1, t2, t3);
        amp = 1.f;
        if (KIND == FAN_SF) {
            const float wx = fmaf((float)i, g.dx, V.o[0]), wy = fmaf((float)j, g.dy, V.o[1]);
            const float r2 = fmaf(wx, wx, wy * wy);
            amp = __fdividef(g.dx * r2 * rsqrtf(r2), fmaxf(fabsf(wx), fabsf(wy)));
        }
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
// contribution of one view's row y to pixel (i, j)
template <typename TIn, int KIND, bool CURVED, bool RECON>
__device__ __forceinline__ float fan_back_view(const CtView &V, const CtGrid &g, const TIn *__restrict__ y, int i,
                                               int j) {
    const float fi = (float)i, fj = (float)j;
    const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
    const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
    if (KIND == FAN_VOX) {
        const float fu = Det<CURVED>::fu(V, cu, cn);
        const float af = floorf(fu), t = fu - af;
        const int a0 = (int)af;
        // cells off the detector weigh zero and read a clamped address
        const float w0 = (a0 >= 0 && a0 < g.nu) ? 1.f - t : 0.f;
        const float w1 = (a0 + 1 >= 0 && a0 + 1 < g.nu) ? t : 0.f;
        const float r = fmaf(w1, ld(y, (size_t)min(max(a0 + 1, 0), g.nu - 1)),
                             w0 * ld(y, (size_t)min(max(a0, 0), g.nu - 1)));
        const float den2 = CURVED ? fmaf(cu, cu, cn * cn) : cn * cn;
        if (RECON) return __fdividef(V.rc_w, den2) * r;
        const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
        const float r2 = fmaf(wx, wx, wy * wy);
        return __fdividef((g.dx * g.dy / g.du) * V.D * r2 * rsqrtf(r2), den2) * r;
    } else if (KIND == FAN_RAY) {
        int aref;
        float fr;
        split_cell(Det<CURVED>::fu(V, cu, cn), aref, fr);
        const float t0 = Det<CURVED>::dfu(V, cu, cn, V.cdu[0], V.cdn[0]);
        const float t1 = Det<CURVED>::dfu(V, cu, cn, V.cdu[1], V.cdn[1]);
        const float t2 = Det<CURVED>::dfu(V, cu, cn, V.cdu[2], V.cdn[2]);
        const float t3 = Det<CURVED>::dfu(V, cu, cn, V.cdu[3], V.cdn[3]);
        const float umin = fr + fminf(fminf(t0, t1), fminf(t2, t3));
        const float umax = fr + fmaxf(fmaxf(t0, t1), fmaxf(t2, t3));
        const int d0 = max((int)ceilf(umin - kSearchPad), -aref);
        const int d1 = min((int)floorf(umax + kSearchPad), g.nu - 1 - aref);
        const float rho = Det<CURVED>::den(cu, cn);
        float s = 0.f;
        for (int d = d0; d <= d1; ++d) {
            const float dfu = (float)d - fr;
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
            if (in && hi > lo) s = fmaf(hi - lo, ld(y, (size_t)(aref + d)), s);
        }
        return s;
    } else {
        Trap T;
        int aref;
        float amp;
        fan_foot<KIND, CURVED>(V, g, i, j, cu, cn, T, aref, amp);
        const int d0 = max((int)floorf(T.k0 + 0.5f), -aref);
        const int d1 = min((int)floorf(T.k3 + 0.5f), g.nu - 1 - aref);
        float s = 0.f, Gp = fan_G<KIND>(T, (float)d0 - 0.5f);
        for (int d = d0; d <= d1; ++d) {
            const float Gn = fan_G<KIND>(T, (float)d + 0.5f);
            s = fmaf(Gn - Gp, ld(y, (size_t)(aref + d)), s);
            Gp = Gn;
        }
        if (RECON) {  // depth weight over the footprint's area (cells) x axial height (rows)
            const float den = Det<CURVED>::den(cu, cn);
            const float area = 0.5f * ((T.k3 - T.k0) + (T.k2 - T.k1));
            amp = __fdividef(V.rc_w, den * V.Kv * fabsf(V.av[2]) * area);
        }
        return amp * s;
    }
}

template <typename TIn, int KIND, bool CURVED, bool RECON>
__global__ void __launch_bounds__(32 * kFanWarps)
fan_back(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ sino, void *__restrict__ vol, int out_t,
         int tiles_x, int batch) {
    __shared__ CtView sview[kFanViews];
    __shared__ float red[kFanWarps][32];
    const int lane = threadIdx.x, w = threadIdx.y, tid = w * 32 + lane;
    const int i = (int)(blockIdx.x % tiles_x) * 8 + (lane & 7), j = (int)(blockIdx.x / tiles_x) * 4 + (lane >> 3);
    const bool active = i < g.nx && j < g.ny;
    for (int bt = blockIdx.y; bt < batch; bt += gridDim.y) {
        const TIn *ys = sino + (size_t)bt * g.nview * g.nu;
        float acc = 0.f;
        for (int v0 = 0; v0 < g.nview; v0 += kFanViews) {
            const int n = min(kFanViews, g.nview - v0);
            __syncthreads();
            const float4 *s4 = reinterpret_cast<const float4 *>(views + v0);
            float4 *d4 = reinterpret_cast<float4 *>(sview);
            for (int t = tid; t < n * (int)(sizeof(CtView) / sizeof(float4)); t += 32 * kFanWarps) d4[t] = __ldg(s4 + t);
            __syncthreads();
            if (active)
                for (int t = w; t < n; t += kFanWarps)
                    acc += fan_back_view<TIn, KIND, CURVED, RECON>(sview[t], g, ys + (size_t)(v0 + t) * g.nu, i, j);
        }
        red[w][lane] = acc;
        __syncthreads();
        if (w == 0 && active) {
            float s = red[0][lane];
#pragma unroll
            for (int q = 1; q < kFanWarps; ++q) s += red[q][lane];
            st_out(g, vol, (size_t)bt * g.ny * g.nx + (size_t)j * g.nx + i, s, out_t);
        }
    }
}

// ------------------------------------------------------------ forward (gather)
// Block = 32 cells of one view.  A warp takes the slabs w, w + 8, ...: the
// pixels of a slab that can reach the tile are evaluated one per lane (weights
// x amplitude x value into the warp's slice of shared memory), then each lane
// adds, for its cell, the pixels between the two lines of constant u that
// bound its footprint's reach (their lateral index is affine in the slab).
template <typename TIn, int KIND, bool CURVED, int NA>
__global__ void __launch_bounds__(32 * kFanWarps)
fan_fwd(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol, void *__restrict__ sino, int out_t,
        int tiles_u) {
    __shared__ CtView V;
    __shared__ float Sw[kFanWarps][NA][32 + 1];
    __shared__ int Sa[kFanWarps][32];
    __shared__ float red[kFanWarps][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    int bx = blockIdx.x;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int v = bx % g.nview;
    const int bt = bx / g.nview;
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
    const TIn *x = vol + (size_t)bt * g.nx * g.ny;
    float acc = 0.f;
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
                const float xv = ld(x, (size_t)j * g.nx + i);
                const float fi = (float)i, fj = (float)j;
                const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
                const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
                if (KIND == FAN_VOX) {
                    const float fu = Det<CURVED>::fu(V, cu, cn);
                    const float af = floorf(fu), t = fu - af;
                    const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
                    const float r2 = fmaf(wx, wx, wy * wy);
                    const float den2 = CURVED ? fmaf(cu, cu, cn * cn) : cn * cn;
                    const float val = __fdividef((g.dx * g.dy / g.du) * V.D * r2 * rsqrtf(r2), den2) * xv;
                    Sw[w][0][lane] = (1.f - t) * val;
                    Sw[w][1][lane] = t * val;
                    Sa[w][lane] = (int)af;
                } else {
                    Trap T;
                    int aref;
                    float amp;
                    fan_foot<KIND, CURVED>(V, g, i, j, cu, cn, T, aref, amp);
                    const int d0 = (int)floorf(T.k0 + 0.5f);
                    const float val = amp * xv;
                    float Gp = 0.f;
#pragma unroll
                    for (int q = 0; q < NA; ++q) {
                        const float Gn = fan_G<KIND>(T, (float)(d0 + q) + 0.5f);
                        Sw[w][q][lane] = (Gn - Gp) * val;
                        Gp = Gn;
                    }
                    Sa[w][lane] = aref + d0;
                }
            }
            __syncwarp();
            const int cb = min(hi, min(base + 31, L1)) - base;
            for (int q = max(lo, base) - base; q <= cb; ++q) {
                const int d = a - Sa[w][q];
                if ((unsigned)d < (unsigned)NA) acc += Sw[w][d][q];
            }
            __syncwarp();
        }
    }
    red[w][lane] = acc;
    __syncthreads();
    if (w || a >= g.nu) return;
    float s = red[0][lane];
#pragma unroll
    for (int q = 1; q < kFanWarps; ++q) s += red[q][lane];
    st_out(g, sino, ((size_t)bt * g.nview + v) * g.nu + a, s * fan_cell_factor<KIND, CURVED>(V, g, a), out_t);
}

// Ray-driven forward: the chord lengths of Siddon's method taken slab by slab
// along the ray's steeper axis (in pixels): the ray's lateral position is
// affine in the slab and moves by at most one pixel across it, so a slab
// meets one pixel, or two that split it at their common edge.  Thread = (ray,
// run of slabs): no serial walk, every slab's loads independent, and the
// sum scaled once by the length of the ray in one slab.
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
    const CtView &V = views[v];
    float cn_ = V.D, cu_ = g.du * ((float)a - V.Cu);
    if (CURVED) {
        float sg, cg;
        sincosf(((float)a - V.Cu) / V.Ku, &sg, &cg);
        cn_ = V.D * cg;
        cu_ = V.D * sg;
    }
    const float d0 = fmaf(cn_, V.nn[0], cu_ * V.eu[0]), d1 = fmaf(cn_, V.nn[1], cu_ * V.eu[1]);
    // source and direction in pixel units; pixel i spans [i - 1/2, i + 1/2)
    const float X0 = -V.o[0] / g.dx, X1 = -V.o[1] / g.dy, D0 = d0 / g.dx, D1 = d1 / g.dy;
    const bool my = fabsf(D1) >= fabsf(D0);  // slabs along y
    const float Sm = my ? X1 : X0, So = my ? X0 : X1, Dm = my ? D1 : D0, Do = my ? D0 : D1;
    const int nm = my ? g.ny : g.nx, no = my ? g.nx : g.ny;
    const int sm = my ? g.nx : 1, so = my ? 1 : g.nx;  // strides of the slab and the lateral index
    const float slope = Do / Dm;
    const float inv = slope != 0.f ? 1.f / slope : 0.f;
    // lateral position at the image's middle (with the slope's rounding taken
    // back over the long way from the source), then slab by slab from there
    const float mid = 0.5f * (float)(nm - 1);
    const float way = mid - Sm;
    const float yc = fmaf(way, slope, So) + way * (fmaf(-slope, Dm, Do) / Dm);
    const TIn *x = vol + (size_t)bt * g.nx * g.ny;
    const int per = (nm + kFanWarps - 1) / kFanWarps;
    const int s0 = w * per, s1 = min(s0 + per, nm);
    float acc = 0.f;
    if (a < g.nu && s0 < s1) {
        float y0 = fmaf((float)s0 - 0.5f - mid, slope, yc);
        int j0 = (int)floorf(y0 + 0.5f);
#pragma unroll 4
        for (int s = s0; s < s1; ++s) {
            const float y1 = fmaf((float)s + 0.5f - mid, slope, yc);
            const int j1 = (int)floorf(y1 + 0.5f);
            const TIn *row = x + (size_t)s * sm;
            const float x0 = (unsigned)j0 < (unsigned)no ? ld(row, (size_t)j0 * so) : 0.f;
            const float x1 = (j1 != j0 && (unsigned)j1 < (unsigned)no) ? ld(row, (size_t)j1 * so) : 0.f;
            // share of the slab before the edge between them
            const float f = j1 == j0 ? 1.f : fminf(fmaxf(((float)max(j0, j1) - 0.5f - y0) * inv, 0.f), 1.f);
            acc = fmaf(f, x0, fmaf(1.f - f, x1, acc));
            y0 = y1;
            j0 = j1;
        }
    }
    red[w][lane] = acc;
    __syncthreads();
    if (w || a >= g.nu) return;
    float s = red[0][lane];
#pragma unroll
    for (int q = 1; q < kFanWarps; ++q) s += red[q][lane];
    s *= sqrtf(fmaf(d0, d0, d1 * d1)) / fabsf(Dm);
    st_out(g, sino, ((size_t)bt * g.nview + v) * g.nu + a, s, out_t);
}

// ------------------------------------------------------------ launchers
namespace {
template <typename TIn, int KIND, bool CURVED>
cudaError_t fan_fwd_k(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                      cudaStream_t st) {
    const int tiles_u = (g.nu + 31) / 32;
    dim3 blk(32, kFanWarps), grd((unsigned)((size_t)tiles_u * g.nview * batch));
    if constexpr (KIND == FAN_RAY) {
        fan_ray_fwd<TIn, CURVED><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    } else if constexpr (KIND == FAN_VOX) {
        fan_fwd<TIn, KIND, CURVED, 2><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    } else {
        // a footprint of half width m meets at most 4 cells when m <= 1.5, 8 when m <= 3.5
        const float m = KIND == FAN_DD ? g.max_m_dd_u : g.max_m_sf_u;
        if (m <= 1.5f)
            fan_fwd<TIn, KIND, CURVED, 4><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
        else
            fan_fwd<TIn, KIND, CURVED, 8><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_u);
    }
    return cudaGetLastError();
}

template <typename TIn, int KIND, bool CURVED, bool RECON>
cudaError_t fan_back_k(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                       cudaStream_t st) {
    const int tiles_x = (g.nx + 7) / 8, tiles_y = (g.ny + 3) / 4;
    dim3 blk(32, kFanWarps), grd((unsigned)tiles_x * (unsigned)tiles_y, (unsigned)std::min(batch, 65535));
    fan_back<TIn, KIND, CURVED, RECON><<<grd, blk, 0, st>>>(g, views, src, out, out_t, tiles_x, batch);
    return cudaGetLastError();
}

template <typename TIn, int KIND>
cudaError_t fan_t(int dir, const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                  cudaStream_t st) {
    const TIn *src = static_cast<const TIn *>(in);
    const bool curved = g.variant == GEO_CIRC_CURVED;
    if (dir == 0)
        return curved ? fan_fwd_k<TIn, KIND, true>(g, views, src, out, out_t, batch, st)
                      : fan_fwd_k<TIn, KIND, false>(g, views, src, out, out_t, batch, st);
    if constexpr (KIND == FAN_SF || KIND == FAN_DD || KIND == FAN_VOX)
        if (dir == 2)
            return curved ? fan_back_k<TIn, KIND, true, true>(g, views, src, out, out_t, batch, st)
                          : fan_back_k<TIn, KIND, false, true>(g, views, src, out, out_t, batch, st);
    return curved ? fan_back_k<TIn, KIND, true, false>(g, views, src, out, out_t, batch, st)
                  : fan_back_k<TIn, KIND, false, false>(g, views, src, out, out_t, batch, st);
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
