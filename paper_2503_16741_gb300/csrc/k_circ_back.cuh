// k_circ_back.cuh -- backprojection in circular cone-beam geometry for the
// projectors whose weight is transaxial x axial: SF-TR, DD and voxel-driven,
// in "proj" and in recon mode (Sec. 2.3; Long, Fessler & Balter 2010; De Man &
// Basu 2004; Peters 1981).
//
// In circular geometry a column's transaxial weights hold for all its voxels,
// and its axial positions are affine in z.  A block owns 32 G columns (8 x 4
// patches, so that a warp's lanes read neighbouring detector cells) and C
// z-chunks of ZT voxels, one (patch, chunk) per warp:
//   set-up:  one thread per (column, view) of a pass of views forms the cell
//            weights, the axial slope and the amplitude factors once for the
//            C chunks that use them (it used to be repeated per chunk, a third
//            of all instructions), into shared memory;
//   filter:  each warp takes every detector row its chunk touches once along
//            u, R(b) = sum_q F[q] y[b][a0 + q], into thread-private shared
//            memory; NT is the host's bound on the cells of a footprint
//            (2 for most DD, 3 for most SF: the loads are what the kernel
//            does most);
//   sweep:   the chunk's voxels walk up those rows.  Consecutive axial
//            rectangles abut, so the walk keeps the distance d from a voxel's
//            lower edge to the next row edge and splits the voxel there.
// Small volumes have fewer (patch, chunk) warps than the chip can hold; the
// blocks of a cluster then share one set of columns, each with every S-th pass
// of views, and add up through distributed shared memory in a fixed order.
// The split depends on the geometry alone: deterministic, and batch items do
// not depend on the batch.
//
// Bound by instruction issue, then L1: the row loads first.
// Measured against the kernels before (set-up per chunk, four taps for every
// footprint, a step-by-step sweep; one column walk per block of views for tall
// voxels), 256^3 / 360 views / 512 x 384 FP32: SF-TR 10.63 -> 7.23 ms, voxel-
// driven recon mode 9.73 -> 5.64 ms; 183^2 x 157 / 231 views, DD with voxels up
// to 1.2 rows high 5.2 -> 1.83 ms; curved 512^2 x 128 / 984 views, DD 50.2 ->
// 31.9 ms; 64^3 / 90 views, DD (views split over 8 blocks) 205 -> 38 us.
#pragma once
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "ct_device.cuh"
#include "ct_launch.h"
#include "k_nc.cuh"

namespace ctp {

namespace cg = cooperative_groups;

namespace {
constexpr int kThreads = 256;  // (column, view) contexts of one pass = threads of a full block

// contexts of one pass
template <int NT> struct BackCtx {
    int as[kThreads];        // first cell read; -1: the column misses the detector; -2 - a (VOX): cell a alone
    int n[kThreads];         // cells with a weight (NT > 4)
    int nw[kThreads];        // the most of them in the warp's 32 columns (NT: cells off the detector among them)
    float F[NT][kThreads];   // their weights (recon: times the depth weight)
    float sv[kThreads];      // rows per voxel
    float fv0[kThreads];     // row of voxel 0's centre
    float im[kThreads];      // amplitude = im sqrt(wz^2 + r2)
    float r2[kThreads];
};
}  // namespace

template <int KIND, bool CURVED, bool RECON, int NT>
__device__ __forceinline__ void back_context(const CtView &V, const CtGrid &g, int i, int j, BackCtx<NT> &S, int t) {
    const float fi = (float)i, fj = (float)j;
    const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
    const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
    const float den2 = CURVED ? fmaf(cu, cu, cn * cn) : cn * cn;
    const float rden = CURVED ? rsqrtf(den2) : rcp_newton(cn);
    const float kd = V.Kv * rden;
    const float sv = kd * V.av[2];
    float F[NT];
    int a0, n;
    float area = 1.f;
    if (KIND == BK_VOX) {
        const float fu = CURVED ? fmaf(V.Ku, atan2f(cu, cn), V.Cu) : fmaf(V.Ku, cu * rden, V.Cu);
        const float af = floorf(fu);
        a0 = (int)af;
        n = 2;
        F[0] = 1.f - (fu - af);
        F[1] = fu - af;
    } else {
        Trap T;
        int aref;
        float k[4];
        column_knots<CURVED, KIND == BK_DD>(V, cu, cn, aref, k);
        const int d0 = (int)floorf(k[0] + 0.5f), d1 = (int)floorf(k[3] + 0.5f);
        a0 = aref + d0;
        if (KIND == BK_DD) {
            T.k0 = T.k1 = k[0];
            T.k2 = T.k3 = k[3];
            T.h1 = T.h3 = 0.f;
#pragma unroll
            for (int q = 0; q < NT; ++q)  // box: plain overlaps
                F[q] = overlap(k[0], k[3], (float)(d0 + q) - 0.5f, (float)(d0 + q) + 0.5f);
            n = min(d1 - d0 + 1, NT);
        } else {
            T = nc_trap(k[0], k[1], k[2], k[3]);
            n = nc_cells<NT>(T, d0, d1, F);
        }
        if (RECON) area = 0.5f * ((k[3] - k[0]) + (k[2] - k[1])) * fabsf(sv);
    }
    if (RECON) {
        const float rw = __fdividef(V.rc_w, den2 * area);
#pragma unroll
        for (int q = 0; q < NT; ++q) F[q] *= rw;
    }
    int as = a0, most = n;
    if (KIND == BK_VOX && (a0 < 0 || a0 + 2 > g.nu)) {  // one of the two cells, or none
        as = a0 == -1 ? -2 : a0 == g.nu - 1 ? -2 - a0 : -1;
        if (a0 == -1) F[0] = F[1];
        F[1] = 0.f;
    } else if (NT > 4 && a0 + NT > g.nu) {  // the cells past the end, which the warp's filter leaves out, dropped
        most = NT;
        n = min(n, g.nu - a0);
        if (n <= 0) as = -1;
    } else if (a0 < 0 || a0 + NT > g.nu) {  // window moved onto the detector, cells off it dropped
        as = min(max(a0, 0), g.nu - NT);
        float Fw[NT];
#pragma unroll
        for (int q = 0; q < NT; ++q) {
            Fw[q] = 0.f;
#pragma unroll
            for (int p = 0; p < NT; ++p)
                if (as + q == a0 + p) Fw[q] = F[p];
        }
#pragma unroll
        for (int q = 0; q < NT; ++q) F[q] = Fw[q];
        if (a0 + n <= 0 || a0 >= g.nu) as = -1;
        most = NT;
        n += min(a0, 0);
    }
    S.as[t] = as;
    if (NT > 4) {
        S.n[t] = n;
        S.nw[t] = __reduce_max_sync(~0u, most);  // (whole warps form contexts)
    }
#pragma unroll
    for (int q = 0; q < NT; ++q) S.F[q][t] = F[q];
    S.sv[t] = sv;
    S.fv0[t] = fmaf(kd, V.av[3], V.Cv);
    if (!RECON && KIND != BK_DD) {
        const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
        S.r2[t] = fmaf(wx, wx, wy * wy);
        S.im[t] = KIND == BK_VOX ? vx_amp(g, V, 1.f, CURVED ? den2 * rden : cn)
                                 : __fdividef(g.dx, fmaxf(fabsf(wx), fabsf(wy)));
    }
}

// A row under the weights that are not zero alone
template <int NT, typename TIn>
__device__ __forceinline__ float own_row(const BackCtx<NT> &X, int t, const TIn *__restrict__ r) {
    float R = 0.f;
#pragma unroll 1
    for (int q = 0; q < NT; ++q) {
        const float f = X.F[q][t];
        if (f != 0.f && (NT <= 4 || q < X.n[t])) R = fmaf(f, ld(r, q), R);
    }
    return R;
}

// The rows r0, r0 + nu, .. (n of them) filtered by a context's first NC weights,
// two rows per step in packed FP32x2 (each lane rounds as the scalar form would).
template <int NC, int NT, typename TIn>
__device__ __forceinline__ void filter_rows(const BackCtx<NT> &X, int t, const TIn *__restrict__ r0, int nu, int n,
                                            float *__restrict__ rw) {
    float2 F2[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) F2[q] = make_float2(X.F[q][t], X.F[q][t]);
    int r = 0;
#pragma unroll 2
    for (; r + 1 < n; r += 2) {
        const TIn *r1 = r0 + nu;
        float2 R = __fmul2_rn(F2[0], make_float2(ld(r0, 0), ld(r1, 0)));
#pragma unroll
        for (int q = 1; q < NC; ++q) R = __ffma2_rn(F2[q], make_float2(ld(r0, q), ld(r1, q)), R);
        rw[0] = R.x;
        rw[kThreads] = R.y;
        rw += 2 * kThreads;
        r0 = r1 + nu;
    }
    if (r < n) {
        float R = F2[0].x * ld(r0, 0);
#pragma unroll
        for (int q = 1; q < NC; ++q) R = fmaf(F2[q].x, ld(r0, q), R);
        rw[0] = R;
    }
}

// NX: rows that a voxel may meet (2: rectangle shorter than a row; 3: than two;
// 5: than four; 9: than eight).  Row buffer: at most ZT sv + 2 rows with
// sv < NX - 1, and the NX rows after them that the last voxel may look at with
// a weight of zero, or of the order of rounding.
// Voxel-driven, voxels of two rows and more (NX > 3): most of the rows between two
// voxels' centres are read by neither, so none is filtered beforehand; each voxel
// filters its own two, and the buffer holds the chunk's sums alone (16 voxels to a
// thread where that leaves the chip a wave of warps, else 4).  342^2 x 292 / 95 views /
// 531 x 2056 FP16: every row filtered 20.5 ms, so 9.1.
__host__ __device__ constexpr bool back_point(int KIND, int NX) { return KIND == BK_VOX && NX > 3; }
__host__ __device__ constexpr int back_rows(int KIND, int ZT, int NX) {
    return back_point(KIND, NX) ? ZT : ZT * (NX - 1) + 2 + NX;
}

template <typename TIn, int KIND, bool CURVED, bool RECON, int NT, int NX, int ZT>
__global__ void __launch_bounds__(kThreads, 4)
circ_back(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ sino, void *__restrict__ vol, int out_t,
          int patches_x, int patches, int C, int nzb, int S) {
    constexpr int NR = back_rows(KIND, ZT, NX);
    constexpr bool POINT = back_point(KIND, NX);
    static_assert(NR >= ZT, "the row buffer also holds the chunk's sums");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BackCtx<NT> *ctx = reinterpret_cast<BackCtx<NT> *>(smem_raw);          // [2]
    float *Rs = reinterpret_cast<float *>(smem_raw + 2 * sizeof(BackCtx<NT>));  // [NR][kThreads]
    const int lane = threadIdx.x, w = threadIdx.y, tid = w * 32 + lane;
    const int G = blockDim.y / C;         // column patches of the block
    const int GC = G * 32, VB = 8 / G;    // columns; views of a pass
    int bx = blockIdx.x;
    const int rank = bx % S; bx /= S;     // cluster rank: the block's share of the passes
    const int zb = bx % nzb; bx /= nzb;
    const int ngrp = (patches + G - 1) / G;
    const int grp = bx % ngrp;
    const int bt = bx / ngrp;
    const int pg = w / C, kbeg = (zb * C + w % C) * ZT;
    const int patch = grp * G + pg;
    const int i = (patch % patches_x) * 8 + (lane & 7), j = (patch / patches_x) * 4 + (lane >> 3);
    const bool active = i < g.nx && j < g.ny && kbeg < g.nz;
    const int len = min(ZT, g.nz - kbeg);
    float acc[ZT];
#pragma unroll
    for (int q = 0; q < ZT; ++q) acc[q] = 0.f;
    const size_t vstride = (size_t)g.nv * g.nu;
    const TIn *ys = sino + (size_t)bt * g.nview * vstride;
    const int npass = (g.nview + VB - 1) / VB;
    auto all_views = [&](auto own) {
        int buf = 0;
        for (int p = rank; p < npass; p += S, buf ^= 1) {
            BackCtx<NT> &X = ctx[buf];
            const int v0 = p * VB, nvc = min(VB, g.nview - v0);
            for (int t = tid; t < nvc * GC; t += blockDim.y * 32) {
                const int c = t % GC, pc = grp * G + (c >> 5);
                const int ci = (pc % patches_x) * 8 + (c & 7), cj = (pc / patches_x) * 4 + ((c & 31) >> 3);
                back_context<KIND, CURVED, RECON, NT>(views[v0 + t / GC], g, ci, cj, X, t);
            }
            // (the other buffer's readers are past the previous pass's barrier)
            __syncthreads();
            if (!active) continue;
            for (int vv = 0; vv < nvc; ++vv) {
                const int t = vv * GC + pg * 32 + lane;
                int as = X.as[t];
                if (as == -1) continue;
                const bool one = KIND == BK_VOX && as < -1;
                if (one) as = -2 - as;
                const float sv = X.sv[t];
                int B;       // first row of the chunk
                float lo;    // the first voxel's lower edge from row B's centre; VOX: its centre from the middle of rows B, B + 1
                int n;       // rows of the chunk
                {
                    int bref;
                    float frac;
                    const float c0 = fmaf(sv, (float)kbeg, X.fv0[t]);
                    if (KIND == BK_VOX) {
                        const float bf = floorf(c0);
                        B = (int)bf;
                        lo = (c0 - bf) - 0.5f;
                        n = (int)floorf(fmaf(sv, (float)(len - 1), lo + 0.5f)) + 2;
                    } else {
                        split_cell(c0, bref, frac);
                        lo = frac - 0.5f * sv;
                        const float ef = floorf(lo + 0.5f);
                        B = bref + (int)ef;
                        lo -= ef;
                        n = (int)ceilf(fmaf(sv, (float)len, lo - 0.5f)) + 1;
                    }
                    n = min(max(n, 0), POINT ? NR : NR - NX);
                }
                const TIn *yp = ys + (size_t)(v0 + vv) * vstride + as;
                if constexpr (POINT) {
                } else if constexpr (decltype(own)::value) {
                    for (int r = 0; r < n; ++r)
                        Rs[r * kThreads + tid] = B + r >= 0 && B + r < g.nv ? own_row(X, t, yp + (size_t)(B + r) * g.nu) : 0.f;
                } else if (B >= 0 && B + n <= g.nv && !one) {
                    const TIn *r0 = yp + (size_t)B * g.nu;
                    // (for NT > 4 the bound holds near the source: most columns need fewer taps)
                    if constexpr (NT <= 4) {
                        filter_rows<NT, NT>(X, t, r0, g.nu, n, Rs + tid);
                    } else if (X.nw[t] <= 3) {
                        filter_rows<3, NT>(X, t, r0, g.nu, n, Rs + tid);
                    } else if (X.nw[t] <= 4) {
                        filter_rows<4, NT>(X, t, r0, g.nu, n, Rs + tid);
                    } else {
                        const int nc = X.n[t];
                        float *rw = Rs + tid;
#pragma unroll 2
                        for (int r = 0; r < n; ++r, r0 += g.nu, rw += kThreads) {
                            float R = X.F[0][t] * ld(r0, 0);
#pragma unroll
                            for (int q = 1; q < NT; ++q)
                                if (q < nc) R = fmaf(X.F[q][t], ld(r0, q), R);
                            rw[0] = R;
                        }
                    }
                } else {  // rows off the detector are zero
                    const int nc = NT > 4 ? X.n[t] : NT;
                    const int second = one ? 0 : 1;  // (one: its cell once more, of weight zero)
                    float *rw = Rs + tid;
                    for (int r = 0; r < n; ++r, rw += kThreads) {
                        const int b = B + r;
                        float R = 0.f;
                        if (b >= 0 && b < g.nv) {
                            const TIn *row = yp + (size_t)b * g.nu;
                            R = X.F[0][t] * ld(row, 0);
#pragma unroll
                            for (int q = 1; q < NT; ++q)
                                if (q < nc) R = fmaf(X.F[q][t], ld(row, KIND == BK_VOX ? second : q), R);
                        }
                        rw[0] = R;
                    }
                }
                if constexpr (!POINT) {
#pragma unroll
                    for (int q = 0; q < NX; ++q) Rs[(n + q) * kThreads + tid] = 0.f;  // (read with weight zero)
                }
                // ---- sweep: voxel kk's lower edge (VOX: centre) lies at p = lo + kk sv rows
                // from row 0's centre (VOX: upper edge); adding 1.5 2^23 rounds p to its row
                // e and leaves e in the low bits, which shifted by 10 are the row's offset
                // in bytes.  Voxels in pairs, in packed FP32x2.
                const char *rp = reinterpret_cast<const char *>(Rs + tid);
                static_assert(kThreads * sizeof(float) == 1 << 10, "row stride of the sweep");
                const float2 sv2 = make_float2(sv, sv), lo2 = make_float2(lo, lo), hi2 = make_float2(0.5f - lo, 0.5f - lo);
                const float2 magic = make_float2(12582912.f, 12582912.f), unmagic = make_float2(-12582912.f, -12582912.f);
                float im = 0.f, r2 = 0.f, wz0 = 0.f;
                if (!RECON && KIND != BK_DD) {
                    im = X.im[t];
                    r2 = X.r2[t];
                    wz0 = fmaf((float)kbeg, g.dz, views[v0 + vv].o[2]);
                }
#pragma unroll
                for (int kk = 0; kk < ZT; kk += 2) {
                    if ((kk & 3) == 0 && kk >= len) break;  // (uniform in the warp; up to 3 voxels past the end are not stored)
                    const float2 k2 = make_float2((float)kk, (float)(kk + 1)), nk2 = make_float2(-(float)kk, -(float)(kk + 1));
                    const float2 m2 = __fadd2_rn(__ffma2_rn(k2, sv2, lo2), magic);
                    // distance from p to the row's upper edge
                    const float2 d2 = __fadd2_rn(__fadd2_rn(m2, unmagic), __ffma2_rn(nk2, sv2, hi2));
                    const char *ra = rp + (int)(__float_as_uint(m2.x) << 10), *rb = rp + (int)(__float_as_uint(m2.y) << 10);
                    auto row = [](const char *r, int q) { return *reinterpret_cast<const float *>(r + q * 1024); };
                    float2 s2;
                    if constexpr (POINT) {
                        auto at = [&](const char *r, int q) {  // that row, filtered here
                            const int b = B + (int)((r - rp) >> 10) + q;
                            if ((unsigned)b >= (unsigned)g.nv) return 0.f;
                            const TIn *y = yp + (size_t)b * g.nu;
                            return fmaf(X.F[1][t], ld(y, one ? 0 : 1), X.F[0][t] * ld(y, 0));
                        };
                        s2 = __fmul2_rn(d2, make_float2(at(ra, 0), at(rb, 0)));
                        s2 = __ffma2_rn(__fadd2_rn(make_float2(1.f, 1.f), make_float2(-d2.x, -d2.y)),
                                        make_float2(at(ra, 1), at(rb, 1)), s2);
                    } else if (KIND == BK_VOX) {  // between rows e and e + 1: d and 1 - d
                        s2 = __fmul2_rn(d2, make_float2(row(ra, 0), row(rb, 0)));
                        s2 = __ffma2_rn(__fadd2_rn(make_float2(1.f, 1.f), make_float2(-d2.x, -d2.y)),
                                        make_float2(row(ra, 1), row(rb, 1)), s2);
                    } else {
                        auto val = [&](const char *r, int q, float f) { return !decltype(own)::value || f > 0.f ? row(r, q) : 0.f; };
                        float2 f2 = make_float2(fminf(d2.x, sv), fminf(d2.y, sv));
                        float2 rest = __fadd2_rn(sv2, make_float2(-f2.x, -f2.y));
                        s2 = __fmul2_rn(f2, make_float2(val(ra, 0, f2.x), val(rb, 0, f2.y)));
#pragma unroll
                        for (int q = 1; q < NX; ++q) {
                            f2 = q + 1 < NX ? make_float2(fminf(rest.x, 1.f), fminf(rest.y, 1.f)) : rest;
                            s2 = __ffma2_rn(f2, make_float2(val(ra, q, f2.x), val(rb, q, f2.y)), s2);
                            if (q + 1 < NX) rest = __fadd2_rn(rest, make_float2(-f2.x, -f2.y));
                        }
                    }
                    float2 amp = make_float2(1.f, 1.f);
                    if (!RECON && KIND != BK_DD) {
                        const float2 wz = make_float2(fmaf((float)kk, g.dz, wz0), fmaf((float)(kk + 1), g.dz, wz0));
                        const float2 q = __ffma2_rn(wz, wz, make_float2(r2, r2));
                        amp = __fmul2_rn(__fmul2_rn(make_float2(im, im), q), make_float2(rsqrtf(q.x), rsqrtf(q.y)));
                    }
                    const float2 a = __ffma2_rn(amp, s2, make_float2(acc[kk], acc[kk + 1]));
                    acc[kk] = a.x;
                    acc[kk + 1] = a.y;
                }
            }
        }
    };
    all_views(std::false_type());
    if constexpr (NX > 2 && KIND != BK_VOX) {
        // Voxels that may be higher than a row: with weights of zero for the rows and
        // cells that a voxel does not meet, an infinite or NaN one among them makes its
        // sum NaN.  A block that has such a sum starts again with these left out (the
        // others come out as before).  In the loops, a test per row or a row of its own
        // in place of each zero cost 6 to 35 % (183^2 x 157 / 231 views DD).
        float bad = 0.f;
#pragma unroll
        for (int kk = 0; kk < ZT; ++kk) bad = kk < len ? fmaf(acc[kk], 0.f, bad) : bad;
        if (__syncthreads_or(active && bad != 0.f)) {
#pragma unroll
            for (int kk = 0; kk < ZT; ++kk) acc[kk] = 0.f;
            all_views(std::true_type());
        }
    }
    const size_t zs = (size_t)g.ny * g.nx;
    const size_t base = ((size_t)bt * g.nz + kbeg) * zs + (size_t)j * g.nx + i;
    if (S == 1) {
        if (!active) return;
#pragma unroll
        for (int kk = 0; kk < ZT; ++kk)
            if (kk < len) st_out(g, vol, base + kk * zs, acc[kk], out_t);
        return;
    }
    // the cluster's sums: rank r stores the voxels r, r + S, ... of every chunk
    cg::cluster_group cl = cg::this_cluster();
#pragma unroll
    for (int kk = 0; kk < ZT; ++kk) Rs[kk * kThreads + tid] = acc[kk];
    cl.sync();
    if (active)
        for (int kk = rank; kk < len; kk += S) {
            float s = 0.f;
            for (int r = 0; r < S; ++r) s += cl.map_shared_rank(Rs, r)[kk * kThreads + tid];
            st_out(g, vol, base + kk * zs, s, out_t);
        }
    cl.sync();  // (a block's shared memory stays until all have read it)
}

// ------------------------------------------------------------ launchers
namespace {
template <typename TIn, int KIND, bool CURVED, bool RECON, int NT, int NX, int ZT>
cudaError_t circ_back_go(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                         cudaStream_t st) {
    const int nch = (g.nz + ZT - 1) / ZT;
    const int nzb = (nch + 7) / 8, C = (nch + nzb - 1) / nzb;  // z-blocks of C <= 8 chunks
    const int G = C == 1 ? 8 : C == 2 ? 4 : C <= 4 ? 2 : 1;
    const int patches_x = (g.nx + 7) / 8, patches = patches_x * ((g.ny + 3) / 4);
    const int ngrp = (patches + G - 1) / G;
    const int npass = (g.nview + 8 / G - 1) / (8 / G);
    const int S = view_split((long long)patches * nch, npass);
    const size_t smem = 2 * sizeof(BackCtx<NT>) + sizeof(float) * back_rows(KIND, ZT, NX) * kThreads;
    auto kern = circ_back<TIn, KIND, CURVED, RECON, NT, NX, ZT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((size_t)S * nzb * ngrp * batch));
    cfg.blockDim = dim3(32, (unsigned)(C * G));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = S > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, g, views, src, out, out_t, patches_x, patches, C, nzb, S);
}

template <typename TIn, int KIND, bool CURVED, bool RECON, int NT>
cudaError_t circ_back_nx(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                         cudaStream_t st) {
    // rows per voxel sv <= 2 max_m_sf_v
    if (g.max_m_sf_v < 0.5f) return circ_back_go<TIn, KIND, CURVED, RECON, NT, 2, 16>(g, views, src, out, out_t, batch, st);
    if (g.max_m_sf_v < 1.f) return circ_back_go<TIn, KIND, CURVED, RECON, NT, 3, 16>(g, views, src, out, out_t, batch, st);
    if constexpr (KIND == BK_VOX) {
        if ((long long)((g.nx + 7) / 8) * ((g.ny + 3) / 4) * ((g.nz + 15) / 16) >= 152 * 32)
            return circ_back_go<TIn, KIND, CURVED, RECON, NT, 9, 16>(g, views, src, out, out_t, batch, st);
    } else if (g.max_m_sf_v < 2.f) {
        return circ_back_go<TIn, KIND, CURVED, RECON, NT, 5, 8>(g, views, src, out, out_t, batch, st);
    }
    return circ_back_go<TIn, KIND, CURVED, RECON, NT, 9, 4>(g, views, src, out, out_t, batch, st);
}

// cells that a footprint of half width m may meet: ceil(2 m) + 1
template <typename TIn, int KIND, bool CURVED, bool RECON>
cudaError_t circ_back_nt(const CtGrid &g, const CtView *views, const TIn *src, void *out, int out_t, int batch,
                         cudaStream_t st) {
    if constexpr (KIND == BK_VOX) {
        return circ_back_nx<TIn, KIND, CURVED, RECON, 2>(g, views, src, out, out_t, batch, st);
    } else {
        const float m = KIND == BK_DD ? g.max_m_dd_u : g.max_m_sf_u;
        if constexpr (KIND == BK_DD)
            if (m <= 0.5f) return circ_back_nx<TIn, KIND, CURVED, RECON, 2>(g, views, src, out, out_t, batch, st);
        if (m <= 1.f) return circ_back_nx<TIn, KIND, CURVED, RECON, 3>(g, views, src, out, out_t, batch, st);
        if (m <= 1.5f) return circ_back_nx<TIn, KIND, CURVED, RECON, 4>(g, views, src, out, out_t, batch, st);
        return circ_back_nx<TIn, KIND, CURVED, RECON, 8>(g, views, src, out, out_t, batch, st);
    }
}

template <typename TIn, int KIND>
cudaError_t circ_back_t(bool recon, const CtGrid &g, const CtView *views, const void *in, void *out, int out_t,
                        int batch, cudaStream_t st) {
    const TIn *src = static_cast<const TIn *>(in);
    const bool curved = g.variant == GEO_CIRC_CURVED;
    if (recon)
        return curved ? circ_back_nt<TIn, KIND, true, true>(g, views, src, out, out_t, batch, st)
                      : circ_back_nt<TIn, KIND, false, true>(g, views, src, out, out_t, batch, st);
    if constexpr (KIND == BK_DD && !std::is_same<TIn, float>::value) return cudaErrorInvalidValue;  // (scaled FP32 only)
    else
        return curved ? circ_back_nt<TIn, KIND, true, false>(g, views, src, out, out_t, batch, st)
                      : circ_back_nt<TIn, KIND, false, false>(g, views, src, out, out_t, batch, st);
}

template <typename TIn>
cudaError_t circ_back_kind(int kind, bool recon, const CtGrid &g, const CtView *views, const void *in, void *out,
                           int out_t, int batch, cudaStream_t st) {
    switch (kind) {
    case BK_SF: return circ_back_t<TIn, BK_SF>(recon, g, views, in, out, out_t, batch, st);
    case BK_DD: return circ_back_t<TIn, BK_DD>(recon, g, views, in, out, out_t, batch, st);
    default: return circ_back_t<TIn, BK_VOX>(recon, g, views, in, out, out_t, batch, st);
    }
}
}  // namespace

}  // namespace ctp
