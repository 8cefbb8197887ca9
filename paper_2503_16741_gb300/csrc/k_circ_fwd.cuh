// k_circ_fwd.cuh -- forward projection in circular cone-beam geometry for the
// projectors whose weight is transaxial x axial: SF-TR, DD and voxel-driven
// (Sec. 2.3; Long, Fessler & Balter 2010; De Man & Basu 2004; Peters 1981).
//
// CTA = 8 to 64 cells x BV = 64, 32 or 8 rows of one view, 256 threads.  Work
// items are the voxel columns (slab s, lateral l) whose footprint can reach the
// tile, taken 256 at a time.
//   stage 1: thread = item; it forms the column's transaxial weights (NT
//            cells, the host's bound) and walks the column, leaving its axial
//            projection onto the tile's rows in shared memory;
//   stage 2: thread = (cell a, RPT rows); it finds, per slab of the round, the
//            items that reach its cell and adds weight x axial projection.
// Each sum has a fixed order: deterministic, and no atomics.  The walk reads a
// copy of the volume in groups of four voxels down z, [z/4][slab][lateral][4],
// one for each main axis that the views have: a warp's load is 32 adjacent columns (512
// contiguous bytes of FP32; in a column-contiguous copy every lane touched a
// cache line of its own, a quarter of the L1 traffic).  The copy pads z with
// zeros, so every height takes the same walk (heights that are no multiple of
// four used to be read voxel by voxel across the slices).
//
// Both stages are bound by instruction issue and the L1/shared pipe.  The walk runs in packed FP32x2: the position of a voxel's edge
// is formed from its index alone (no chain from voxel to voxel), rounded to its
// row by adding 1.5 2^23, whose low bits then are the row's offset in shared
// memory; a closed row is stored by one predicated instruction (as a branch it
// cost a quarter of the kernel: 120 views of the 256^3 scan 5.5 -> 4.3 ms), and
// the next four voxels are requested before the present ones are walked (the
// curved scan below: 83 -> 50 ms, with three blocks per SM instead of two).
// Of the 256^3 scan's time (11.4 ms before the 64-cell tiles), compiling parts
// out left: set-up and search 1.3 ms, walk 5.6, stage 2 5.0.
// Measured against the kernel before, 256^3 / 360 views / 512 x 384 FP32: SF-TR
// 13.4 -> 10.6 ms, voxel-driven 19.2 -> 10.2 ms; 161^2 x 155 / 607 views, SF-TR
// 10.4 -> 5.1 ms (no multiple of four slices); 183^2 x 157 / 231 views, DD with
// voxels up to 1.2 rows high 6.4 -> 3.7 ms; curved 512^2 x 128 / 984 views, DD
// 65.3 -> 48 ms.
#pragma once
#include <algorithm>

#include "ct_device.cuh"
#include "ct_launch.h"
#include "k_nc.cuh"

namespace ctp {

// CTAs of tiles `cells` wide and 64 rows high, and a wave of them (three to an SM)
inline long long circ_fwd_ctas(const CtGrid &g, int cells, int batch) {
    return (long long)((g.nu + cells - 1) / cells) * ((g.nv + 63) / 64) * g.nview * batch;
}
constexpr long long kFwdWave = 3 * 152;
// What the kernel reads: the copies (nzp > 0: slices of one; see circ_fwd) or, nzp = 0,
// the volume in place, which gives the same results, slower where the copies pay
struct FwdVolume {
    const void *y, *x;
    int nzp;
};
// The smallest volumes are read in place in calls of few CTAs: the copies would cost
// such a call an allocation and a launch, a third of its time.
inline bool circ_fwd_direct(const CtGrid &g, int batch) {
    return !copies_pay(g, batch) && circ_fwd_ctas(g, 32, batch) < kFwdWave;
}

namespace {
constexpr int kFwdItems = 256;  // items of a round = threads
constexpr int kFwdSeg = 256;    // slabs of a segment

template <int BV, int NT> struct CircFwdSmem {
    float Z[BV][kFwdItems];  // [row][item]
    // the item's transaxial weights x amplitude factor; rows padded by 8 so that
    // lanes reading one item's weights of different cells fall on different banks
    float Fu[NT][kFwdItems + 8];
    short a0[kFwdItems + 2];  // first cell of the item's weights, from the tile's first cell
    unsigned short L0[kFwdSeg];  // first column of each slab (at most 65536 columns)
    int off[kFwdSeg + 1];        // first item of each slab
    int warp_sum[8];
};
}  // namespace

// Voxels k .. k + 3 of a column from the address of voxel k: four in a row in a
// copy, which is padded with zeros, or (DIRECT) a slice apart in the volume itself.
template <bool DIRECT, typename TIn>
__device__ __forceinline__ void walk_load(const CtGrid &g, const TIn *__restrict__ p, int k, float (&x)[4]) {
    if constexpr (DIRECT) {
        const size_t zs = (size_t)g.nx * g.ny;
#pragma unroll
        for (int t = 0; t < 4; ++t) x[t] = k + t < g.nz ? ld(p, t * zs) : 0.f;
    } else {
        ld4(p, x);
    }
}

// Stage 1's walk.  Voxel k's rectangle covers rows [p, p + sv] with p = lo +
// (k - ks) sv (rows from the tile's row 0; VOX: p is its centre's row minus one
// half), and consecutive rectangles abut, so every row's sum is complete when
// a voxel's upper edge lies in another row, and is stored once.  (Whether it
// does is read off the rounded edge that the next voxel starts from, so the
// two agree whatever the rounding.)  TALL: a voxel may cover whole rows.
// Voxels outside [k0, k1] reach no row of the tile.
template <typename TIn, int KIND, int BV, bool TALL, bool DIRECT>
__device__ __forceinline__ void circ_walk(const CtGrid &g, const TIn *__restrict__ cz, size_t pitch, float (&xa)[4],
                                          int k0, int k1, float sv, float fv0, float r2, float oz, int B0,
                                          float (&Z)[BV][kFwdItems], int tid) {
    static_assert(kFwdItems * sizeof(float) == 1 << 10, "row stride of the walk");
    const int ks = k0 & ~3;
    float lo;  // of voxel ks
    {
        int bref;
        float frac;
        split_cell(fmaf(sv, (float)ks, fv0), bref, frac);
        lo = (frac - (KIND == BK_VOX ? 0.5f : 0.5f * sv)) + (float)(bref - B0);
    }
    const float2 magic = make_float2(12582912.f, 12582912.f), minus1 = make_float2(-1.f, -1.f);
    const float2 sv2 = make_float2(sv, sv);
    const float wz0 = fmaf((float)ks, g.dz, oz);
    // rows below the walk's first one
    int open = (int)(__float_as_uint(lo + 12582912.f) << 10);  // byte offset of the open row
    // (VOX: rows between two voxels' rows, which the walk passes over)
    for (int q = 0; q < (TALL && KIND == BK_VOX && sv > 1.9f ? BV : min(open >> 10, BV)); ++q) Z[q][tid] = 0.f;
    float acc = 0.f, acc1 = 0.f;  // sum of the open row (VOX: and of the next)
    const unsigned zt = (unsigned)__cvta_generic_to_shared(&Z[0][tid]);
    auto put = [&](int off, float v) {  // into the tile's rows only
        asm volatile("{ .reg .pred q; setp.lt.u32 q, %0, %1; @q st.shared.f32 [%2], %3; }" ::"r"(off), "n"(BV << 10),
                     "r"(zt + off), "f"(v)
                     : "memory");
    };
    // the same when the row changes from `off` to `next` (one predicated store, no branch)
    auto put_if = [&](int off, int next, float v) {
        asm volatile(
            "{ .reg .pred p, q; setp.ne.s32 p, %0, %4; setp.lt.and.u32 q, %0, %1, p; @q st.shared.f32 [%2], %3; }" ::"r"(off),
            "n"(BV << 10), "r"(zt + off), "f"(v), "r"(next)
            : "memory");
    };
    // the same when the row `next` lies above `off`
    auto put_above = [&](int off, int next, float v) {
        asm volatile(
            "{ .reg .pred p, q; setp.lt.s32 p, %0, %4; setp.lt.and.u32 q, %0, %1, p; @q st.shared.f32 [%2], %3; }" ::"r"(off),
            "n"(BV << 10), "r"(zt + off), "f"(v), "r"(next)
            : "memory");
    };
    // voxels kk .. kk + 3 of the walk (kk from ks)
    auto quad = [&](float kk, const float *x4) {
        const float pq = fmaf(kk, sv, lo), ph = pq + 0.5f, wk = fmaf(kk, g.dz, wz0);
#pragma unroll
        for (int t = 0; t < 4; t += 2) {
            // upper edges of the two voxels (VOX: their centres)
            constexpr float kUp = KIND == BK_VOX ? 0.f : 1.f;
            const float2 k2 = make_float2((float)t + kUp, (float)(t + 1) + kUp);
            const float2 m2 = __fadd2_rn(__ffma2_rn(k2, sv2, make_float2(pq, pq)), magic);
            // their distance from the row's lower edge
            const float2 w2 = __fadd2_rn(__ffma2_rn(k2, sv2, make_float2(ph, ph)), __ffma2_rn(m2, minus1, magic));
            float2 v2 = make_float2(x4[t], x4[t + 1]);
            if (KIND != BK_DD) {  // times the distance to the source (its factor is in the transaxial weights)
                const float2 wz = make_float2(fmaf((float)t, g.dz, wk), fmaf((float)(t + 1), g.dz, wk));
                const float2 q = __ffma2_rn(wz, wz, make_float2(r2, r2));
                v2 = __fmul2_rn(__fmul2_rn(q, make_float2(rsqrtf(q.x), rsqrtf(q.y))), v2);
            }
            if constexpr (KIND == BK_VOX) {  // w to the row above, 1 - w to the row (v - w v would be NaN for an infinite v)
                const float2 up2 = __fmul2_rn(w2, v2), own2 = __fmul2_rn(__ffma2_rn(w2, minus1, make_float2(1.f, 1.f)), v2);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int off = (int)(__float_as_uint(h ? m2.y : m2.x) << 10);
                    put_if(open, off, acc);
                    if (TALL) {  // the centre may pass rows
                        const int next = open + (1 << 10);
                        put_above(next, off, acc1);
                        acc1 = off > next ? 0.f : acc1;
                    }
                    acc = off != open ? acc1 : acc;
                    acc1 = off != open ? 0.f : acc1;
                    open = off;
                    acc += h ? own2.y : own2.x;
                    acc1 += h ? up2.y : up2.x;
                }
            } else {
                // the part in the row of the upper edge, and the part below it
                const float2 g2 = make_float2(fminf(w2.x, sv), fminf(w2.y, sv));
                const float2 f2 = __ffma2_rn(g2, minus1, sv2);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float v = h ? v2.y : v2.x, gv = h ? g2.y : g2.x;
                    float f = h ? f2.y : f2.x;
                    const int off = (int)(__float_as_uint(h ? m2.y : m2.x) << 10);
                    const bool cross = off != open;
                    if (!TALL) {
                        put_if(open, off, fmaf(f, v, acc));
                    } else if (cross) {  // rows wholly inside the voxel
                        const int first = open;
                        f -= (float)((off - open >> 10) - 1);
                        for (int o = open + (1 << 10); o < off; o += 1 << 10) put(o, v);
                        put(first, fmaf(f, v, acc));
                    }
                    acc = fmaf(gv, v, cross ? 0.f : acc);
                    open = off;
                }
            }
        }
    };
    // four voxels per load, the next four requested before they are walked
    // (xa: the first four, requested by the caller)
    const TIn *cq = cz + (size_t)(ks >> 2) * pitch;
    float xb[4];
    float kk = 0.f;
    for (int left = k1 - ks, k = ks + 4;; left -= 8, k += 8, kk += 8.f) {
        if (left >= 4) walk_load<DIRECT>(g, cq + pitch, k, xb);
        quad(kk, xa);
        if (left < 4) break;
        cq += 2 * pitch;
        if (left >= 8) walk_load<DIRECT>(g, cq, k + 4, xa);
        quad(kk + 4.f, xb);
        if (left < 8) break;
    }
    put(open, acc);
    int r = (open >> 10) + 1;
    if (KIND == BK_VOX) {
        put(open + (1 << 10), acc1);
        ++r;
    }
    for (int q = max(r, 0); q < BV; ++q) Z[q][tid] = 0.f;
}

// CTA = CELLS cells x BV rows, RPT rows to a thread, NG threads to a cell.
// (BV = 64: 3 blocks per SM by shared memory and 80 registers; 32 x 32: 4 at 64)
// vol_y, vol_x: the copies for the views whose main axis is y and x; null: not these
// views.  DIRECT: the volume itself instead.
template <typename TIn, int KIND, bool CURVED, int CELLS, int BV, int NT, bool TALL, bool DIRECT>
__global__ void __launch_bounds__(256, BV == 64 ? 3 : 4)
circ_fwd(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol_y, const TIn *__restrict__ vol_x, int nzp,
         void *__restrict__ sino, int out_t, int tiles_u, int tiles_v) {
    constexpr int NG = 256 / CELLS, RPT = BV / NG;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CircFwdSmem<BV, NT> &S = *reinterpret_cast<CircFwdSmem<BV, NT> *>(smem_raw);
    int bx = blockIdx.x;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int tv = bx % tiles_v; bx /= tiles_v;
    const int v = bx % g.nview;
    const int bt = bx / g.nview;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int A0 = tu * CELLS, B0 = tv * BV, Bn = min(BV, g.nv - B0);  // rows of the tile on the detector
    // the thread's cell in the tile, and its rows rg, rg + NG, ..
    const int ac = CELLS == 32 ? (int)threadIdx.x : tid % CELLS, rg = CELLS == 32 ? (int)threadIdx.y : tid / CELLS;
    const int a = A0 + ac;
    const CtView &V = views[v];
    const int main_y = V.main_y;
    const TIn *xz = main_y ? vol_y : vol_x;
    if (!xz) return;  // (whole CTA)
    const SlabCoef sc = slab_coef(V, main_y);
    // search half widths: footprint bound + half a cell, or the hat's one cell
    const float mu = KIND == BK_VOX ? 1.f + kSearchPad : (KIND == BK_DD ? V.m_dd_u : V.m_sf_u) + 0.5f + kSearchPad;
    const float mv = KIND == BK_VOX ? 1.f + kSearchPad : V.m_sf_v + 0.5f + kSearchPad;
    const int nslab = main_y ? g.ny : g.nx, nlat = main_y ? g.nx : g.ny;
    // the copy whose columns are adjacent along the view's lateral axis
    xz += (size_t)bt * (DIRECT ? g.nz : nzp) * g.nx * g.ny;
    // the two lines of constant u that bound the cell's reach: lateral index = p + s slab
    float p1, s1, p2, s2;
    {
        const float T1 = Det<CURVED>::ratio_at(V, a - mu), T2 = Det<CURVED>::ratio_at(V, a + mu);
        const float q1 = 1.f / (sc.ul - T1 * sc.nl), q2 = 1.f / (sc.ul - T2 * sc.nl);
        p1 = fmaf(T1, sc.n3, -sc.u3) * q1;
        s1 = fmaf(T1, sc.ns, -sc.us) * q1;
        p2 = fmaf(T2, sc.n3, -sc.u3) * q2;
        s2 = fmaf(T2, sc.ns, -sc.us) * q2;
    }
    float2 acc[(RPT + 1) / 2];
#pragma unroll
    for (int r = 0; r < (RPT + 1) / 2; ++r) acc[r] = make_float2(0.f, 0.f);

    for (int seg = 0; seg < nslab; seg += kFwdSeg) {
        const int nseg = min(kFwdSeg, nslab - seg);
        // column range of every slab of the segment for the whole tile
        __syncthreads();
        int c = 0;
        if (tid < nseg) {
            int L0, L1, K0, K1;
            if (slab_search<CURVED>(V, sc, seg + tid, A0 - mu, A0 + (CELLS - 1.f) + mu, B0 - mv, B0 + Bn - 1.f + mv, nlat, g.nz,
                                    L0, L1, K0, K1))
                c = L1 - L0 + 1;
            S.L0[tid] = (unsigned short)(c ? L0 : 0);
        }
        {  // exclusive prefix sum over the segment
            int o = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(~0u, o, d);
                if ((tid & 31) >= d) o += u;
            }
            if ((tid & 31) == 31) S.warp_sum[tid >> 5] = o;
            __syncthreads();
            for (int w = 0; w < (tid >> 5); ++w) o += S.warp_sum[w];
            if (tid < nseg) S.off[tid + 1] = o;
            if (tid == 0) S.off[0] = 0;
        }
        __syncthreads();
        const int total = S.off[nseg];
        // last slab t' >= t with off[t'] <= q, by the whole warp: 32 offsets at a time
        auto seek = [&](int t, int q) {
            for (;;) {
                const int u = t + 1 + (int)threadIdx.x;
                const int c = __popc(__ballot_sync(~0u, u < nseg && S.off[min(u, nseg)] <= q));
                t += c;
                if (c < 32) return t;
            }
        };
        int first = 0;  // slab of the round's first item
        for (int base = 0; base < total; base += kFwdItems) {
            // ---- stage 1: one item (column) per thread
            const int q = base + tid;
            first = seek(first, base);
            int lo = seek(first, base + (tid & ~31));  // slab of the warp's first item
            if (q < total) {
                // each lane steps forward to its own item's slab (a slab holds tens of items)
                while (lo < nseg - 1 && S.off[lo + 1] <= q) ++lo;
                const int s = seg + lo;
                const int l = S.L0[lo] + (q - S.off[lo]);
                const int i = main_y ? l : s, j = main_y ? s : l;
                const float fi = (float)i, fj = (float)j;
                const float cu = fmaf(V.au[0], fi, fmaf(V.au[1], fj, V.au[3]));
                const float cn = fmaf(V.an[0], fi, fmaf(V.an[1], fj, V.an[3]));
                const float den2 = CURVED ? fmaf(cu, cu, cn * cn) : cn * cn;
                const float rden = CURVED ? rsqrtf(den2) : rcp_newton(cn);
                const float kd = V.Kv * rden;
                const float sv = kd * V.av[2], fv0 = fmaf(kd, V.av[3], V.Cv);
                const float wx = fmaf(fi, g.dx, V.o[0]), wy = fmaf(fj, g.dy, V.o[1]);
                // voxels that can meet a row of the tile
                const float hw = KIND == BK_VOX ? 1.f + kSearchPad : 0.5f + 0.5f * sv + kSearchPad;
                const float rsv = __fdividef(1.f, sv);
                const int k0 = max(0, (int)ceilf(((float)B0 - fv0 - hw) * rsv - 1e-3f));
                const int k1 = min(g.nz - 1, (int)floorf(((float)(B0 + Bn - 1) - fv0 + hw) * rsv + 1e-3f));
                const TIn *cz = xz + (DIRECT ? (size_t)j * g.nx + i : 4 * ((size_t)s * nlat + l));
                const size_t pitch = 4 * (size_t)g.nx * g.ny;
                float x4[4] = {0.f, 0.f, 0.f, 0.f};  // on its way while the weights are formed
                if (k0 <= k1) walk_load<DIRECT>(g, cz + (size_t)(k0 >> 2) * pitch, k0 & ~3, x4);
                if constexpr (KIND == BK_VOX) {
                    const float fu = CURVED ? fmaf(V.Ku, atan2f(cu, cn), V.Cu) : fmaf(V.Ku, cu * rden, V.Cu);
                    const float af = floorf(fu), amp = vx_amp(g, V, 1.f, CURVED ? den2 * rden : cn);
                    S.Fu[0][tid] = (1.f - (fu - af)) * amp;
                    S.Fu[1][tid] = (fu - af) * amp;
                    S.a0[tid] = (short)((int)af - A0);
                } else {
                    int aref;
                    float kn[4], F[NT];
                    column_knots<CURVED, KIND == BK_DD>(V, cu, cn, aref, kn);
                    const int d0 = (int)floorf(kn[0] + 0.5f), d1 = (int)floorf(kn[3] + 0.5f);
                    if (KIND == BK_DD) {
#pragma unroll
                        for (int r = 0; r < NT; ++r)
                            F[r] = overlap(kn[0], kn[3], (float)(d0 + r) - 0.5f, (float)(d0 + r) + 0.5f);
                    } else {
                        const Trap T = nc_trap(kn[0], kn[1], kn[2], kn[3]);
                        nc_cells<NT>(T, d0, d1, F);
                        const float im = __fdividef(g.dx, fmaxf(fabsf(wx), fabsf(wy)));
#pragma unroll
                        for (int r = 0; r < NT; ++r) F[r] *= im;
                    }
#pragma unroll
                    for (int r = 0; r < NT; ++r) S.Fu[r][tid] = F[r];
                    S.a0[tid] = (short)(aref + d0 - A0);
                }
                if (k0 <= k1)
                    circ_walk<TIn, KIND, BV, TALL, DIRECT>(g, cz, pitch, x4, k0, k1, sv, fv0, fmaf(wx, wx, wy * wy),
                                                           V.o[2], B0, S.Z, tid);
                else
                    for (int r = 0; r < BV; ++r) S.Z[r][tid] = 0.f;
            }
            __syncthreads();
            // ---- stage 2: thread = (cell a, rows B0 + rg + NG r)
            if (a < g.nu) {
                const int qend = min(total, base + kFwdItems);
                const float *zr = &S.Z[rg][0];
                for (int t = first, o0 = S.off[first]; t < nseg && o0 < qend; ++t) {
                    const int o1 = S.off[t + 1];
                    const float fs = (float)(seg + t);
                    const float la = fmaf(s1, fs, p1), lb = fmaf(s2, fs, p2);
                    // items of the slab in this round that reach the cell (1e-3 column: rounding of the lines)
                    const int rel = o0 - base - S.L0[t];
                    const int c0 = max((int)ceilf(fminf(la, lb) - 1e-3f) + rel, max(o0 - base, 0));
                    const int c1 = min((int)floorf(fmaxf(la, lb) + 1e-3f) + rel, min(o1, qend) - base - 1);
                    o0 = o1;
                    if (c0 > c1) continue;
                    for (int c = c0, next = S.a0[c0]; c <= c1; ++c) {
                        const int d = ac - next;
                        next = S.a0[c + 1];  // (the next item's, before this one's rows)
                        if ((unsigned)d >= (unsigned)NT) continue;
                        const float w = S.Fu[d][c];
                        const float *z = zr + c;
                        if constexpr (RPT % 2 == 0) {  // row pairs in packed FP32x2
                            const float2 w2 = make_float2(w, w);
#pragma unroll
                            for (int r = 0; r < RPT; r += 2)
                                acc[r / 2] = __ffma2_rn(w2, make_float2(z[NG * r * kFwdItems], z[NG * (r + 1) * kFwdItems]),
                                                        acc[r / 2]);
                        } else {
                            acc[0].x = fmaf(w, z[0], acc[0].x);
                        }
                    }
                }
            }
            __syncthreads();
        }
    }
    if (a < g.nu) {
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int b = B0 + rg + NG * r;
            const float s = (r & 1) ? acc[r / 2].y : acc[r / 2].x;
            if (b < g.nv)
                st_out(g, sino, (((size_t)bt * g.nview + v) * g.nv + b) * g.nu + a,
                       KIND == BK_DD ? s * dd_len<CURVED>(V, g, a, b) : s, out_t);
        }
    }
}

// ------------------------------------------------------------ launchers
namespace {
template <typename TIn, int KIND, bool CURVED, int CELLS, int BV, int NT, bool TALL, bool DIRECT = false>
cudaError_t circ_fwd_go(const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t, int batch,
                        cudaStream_t st) {
    const int tiles_u = (g.nu + CELLS - 1) / CELLS, tiles_v = (g.nv + BV - 1) / BV;
    const size_t smem = sizeof(CircFwdSmem<BV, NT>);
    auto kern = circ_fwd<TIn, KIND, CURVED, CELLS, BV, NT, TALL, DIRECT>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((unsigned)((size_t)tiles_u * tiles_v * g.nview * batch)), dim3(32, 8), smem, st>>>(
        g, views, static_cast<const TIn *>(x.y), static_cast<const TIn *>(x.x), x.nzp, out, out_t, tiles_u, tiles_v);
    return cudaGetLastError();
}

// The tile.  Its height follows the detector alone, since a column's walk starts
// where the tile does: 64 rows, or fewer where they hold the detector (which leaves
// the walk as it is).  64 even for a detector that is cut into few tiles: a column's
// set-up is shared by twice the rows of a 32-row tile (64^3 / 360 views / 128 x 96
// SF-TR 452 -> 353 us, curved 256^2 x 64 / 246 views / 444 x 64 DD 3813 -> 3040 us);
// 8 for a short one (96^2 x 8 / 143 views / 150 x 4 SF-TR 178 -> 127 us against 32).
// Its width decides how many CTAs there are and changes no bit of a result, so it
// may follow the views and the batch.  64 cells are the fastest where they fill the
// chip: a thread of stage 2 sums 16 rows and shares what it does per column among
// them (256^3 / 360 views SF-TR 11.4 -> 10.5 ms against 32).  But a CTA takes the time
// of its columns in all slabs, however few others run: below two waves (three CTAs to
// an SM) 32 cells, below one 16, below a quarter 8.  256^3 / 512 x 384 SF-TR, 64, 32
// and 16 cells: 1 view 1147, 509, 320 us; 8 views 1143, 653, 574; 16 views 1138, 829,
// 859; 32 views 1462, 1304, 1441; 64 views 2360, 2312, 2687.  64^3 / 1 view / 128 x 96
// DD, 16 and 8 cells: 59, 49 us.  (16 rows by 16 cells in their place: better for one
// view, up to twice the time for a few.)  Voxels that may cover whole rows have a walk
// that spills at 64 x 64 (183^2 x 157 / 231 views DD 3.7 -> 4.2 ms).
template <typename TIn, int KIND, bool CURVED, int NT, bool TALL>
cudaError_t circ_fwd_rpt(const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t, int batch,
                         cudaStream_t st) {
    // (TALL everywhere: one kernel serves either height of voxels in small calls and in place)
    if (x.nzp == 0) {
        if (g.nv <= 8) return circ_fwd_go<TIn, KIND, CURVED, 32, 8, NT, true, true>(g, views, x, out, out_t, batch, st);
        if (circ_fwd_ctas(g, 32, batch) < kFwdWave)
            return circ_fwd_go<TIn, KIND, CURVED, 16, 64, NT, true, true>(g, views, x, out, out_t, batch, st);
        return circ_fwd_go<TIn, KIND, CURVED, 32, 64, NT, true, true>(g, views, x, out, out_t, batch, st);
    }
    if (g.nv <= 8) return circ_fwd_go<TIn, KIND, CURVED, 32, 8, NT, true>(g, views, x, out, out_t, batch, st);
    if (circ_fwd_ctas(g, 16, batch) < kFwdWave / 2)
        return circ_fwd_go<TIn, KIND, CURVED, 8, 64, NT, true>(g, views, x, out, out_t, batch, st);
    if (circ_fwd_ctas(g, 32, batch) < kFwdWave)
        return circ_fwd_go<TIn, KIND, CURVED, 16, 64, NT, TALL>(g, views, x, out, out_t, batch, st);
    if (g.nv <= 32) return circ_fwd_go<TIn, KIND, CURVED, 32, 32, NT, TALL>(g, views, x, out, out_t, batch, st);
    if constexpr (!TALL)
        if (circ_fwd_ctas(g, 64, batch) >= 2 * kFwdWave)
            return circ_fwd_go<TIn, KIND, CURVED, 64, 64, NT, TALL>(g, views, x, out, out_t, batch, st);
    return circ_fwd_go<TIn, KIND, CURVED, 32, 64, NT, TALL>(g, views, x, out, out_t, batch, st);
}

template <typename TIn, int KIND, bool CURVED, int NT>
cudaError_t circ_fwd_nx(const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t, int batch,
                        cudaStream_t st) {
    // rows per voxel: at most 2 max_m_sf_v
    if (g.max_m_sf_v < 0.5f) return circ_fwd_rpt<TIn, KIND, CURVED, NT, false>(g, views, x, out, out_t, batch, st);
    return circ_fwd_rpt<TIn, KIND, CURVED, NT, true>(g, views, x, out, out_t, batch, st);
}

template <typename TIn, int KIND, bool CURVED>
cudaError_t circ_fwd_nt(const CtGrid &g, const CtView *views, const FwdVolume &x, void *out, int out_t, int batch,
                        cudaStream_t st) {
    if constexpr (KIND == BK_VOX) {
        return circ_fwd_nx<TIn, KIND, CURVED, 2>(g, views, x, out, out_t, batch, st);
    } else {
        // cells that a footprint of half width m may meet: ceil(2 m) + 1
        const float m = KIND == BK_DD ? g.max_m_dd_u : g.max_m_sf_u;
        if (m <= 1.f) return circ_fwd_nx<TIn, KIND, CURVED, 3>(g, views, x, out, out_t, batch, st);
        if (m <= 1.5f) return circ_fwd_nx<TIn, KIND, CURVED, 4>(g, views, x, out, out_t, batch, st);
        if (m <= 2.5f) return circ_fwd_nx<TIn, KIND, CURVED, 6>(g, views, x, out, out_t, batch, st);
        return circ_fwd_nx<TIn, KIND, CURVED, 8>(g, views, x, out, out_t, batch, st);
    }
}

template <typename TIn>
cudaError_t circ_fwd_kind(int kind, const CtGrid &g, const CtView *views, const FwdVolume &x, void *out,
                          int out_t, int batch, cudaStream_t st) {
    const bool curved = g.variant == GEO_CIRC_CURVED;
    switch (kind) {
    case BK_SF:
        return curved ? circ_fwd_nt<TIn, BK_SF, true>(g, views, x, out, out_t, batch, st)
                      : circ_fwd_nt<TIn, BK_SF, false>(g, views, x, out, out_t, batch, st);
    case BK_DD:
        return curved ? circ_fwd_nt<TIn, BK_DD, true>(g, views, x, out, out_t, batch, st)
                      : circ_fwd_nt<TIn, BK_DD, false>(g, views, x, out, out_t, batch, st);
    default:
        return curved ? circ_fwd_nt<TIn, BK_VOX, true>(g, views, x, out, out_t, batch, st)
                      : circ_fwd_nt<TIn, BK_VOX, false>(g, views, x, out, out_t, batch, st);
    }
}
}  // namespace

}  // namespace ctp
