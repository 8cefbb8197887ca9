// k_nc_fwd.cu -- forward projection of the non-circular SF-TR and DD
// footprint projectors and of SF-TT (the footprint and the dispatch are in
// k_nc.cuh).
#include "k_nc.cuh"

namespace ctp {

// ------------------------------------------------------------ forward (gather)
// Index box of slab s for a detector window [Flo, Fhi] x [Glo, Ghi]: the
// window's four corner rays meet the slab plane at points whose lateral and
// axial indices are affine in s (the plane equations are affine in s and
// their 2 x 2 determinant does not depend on s), so the box of every slab
// comes from 8 coefficient pairs formed once per thread.
struct NcBox {
    float l0[4], l1[4], k0[4], k1[4];  // l = l0 + l1 s, k = k0 + k1 s per corner ray
};

__device__ __forceinline__ NcBox nc_box_coef(const CtView &V, const SlabCoef &c, float Flo, float Fhi,
                                             float Glo, float Ghi) {
    NcBox B;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float tu = (q ? Fhi : Flo) - V.Cu;
        const float Pl = fmaf(V.Ku, c.ul, -tu * c.nl);
        const float Pk = fmaf(V.Ku, c.uk, -tu * c.nk);
        const float P0 = fmaf(V.Ku, c.u3, -tu * c.n3), P1 = fmaf(V.Ku, c.us, -tu * c.ns);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float tv = (r ? Ghi : Glo) - V.Cv;
            const float Ql = fmaf(V.Kv, c.vl, -tv * c.nl);
            const float Qk = fmaf(V.Kv, c.vk, -tv * c.nk);
            const float Q0 = fmaf(V.Kv, c.v3, -tv * c.n3), Q1 = fmaf(V.Kv, c.vs, -tv * c.ns);
            const float rdet = 1.f / fmaf(Pl, Qk, -Pk * Ql);
            const int t = 2 * q + r;
            B.l0[t] = fmaf(-P0, Qk, Q0 * Pk) * rdet;
            B.l1[t] = fmaf(-P1, Qk, Q1 * Pk) * rdet;
            B.k0[t] = fmaf(-Q0, Pl, P0 * Ql) * rdet;
            B.k1[t] = fmaf(-Q1, Pl, P1 * Ql) * rdet;
        }
    }
    return B;
}

__device__ __forceinline__ bool nc_box(const NcBox &B, float s, int nlat, int nk, int &l0, int &l1, int &k0,
                                       int &k1) {
    float lmin = 3.0e38f, lmax = -3.0e38f, kmin = 3.0e38f, kmax = -3.0e38f;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float l = fmaf(B.l1[t], s, B.l0[t]), k = fmaf(B.k1[t], s, B.k0[t]);
        lmin = fminf(lmin, l); lmax = fmaxf(lmax, l);
        kmin = fminf(kmin, k); kmax = fmaxf(kmax, k);
    }
    if (!(isfinite(lmin) && isfinite(lmax) && isfinite(kmin) && isfinite(kmax))) return false;
    l0 = max(0, (int)ceilf(lmin));
    l1 = min(nlat - 1, (int)floorf(lmax));
    k0 = max(0, (int)ceilf(kmin));
    k1 = min(nk - 1, (int)floorf(kmax));
    return l0 <= l1 && k0 <= k1;
}

// Footprint cache of one round: per voxel its NA transaxial weights times
// amplitude times value, its axial weights placed in an 8-row window that
// starts at a 4-row group boundary of the tile, and (first cell, group).
// Lateral index at which a line of constant fu meets row k of slab s:
// l = c0 + ck k + cs s (the line Ku (au.X) = (F - Cu) (an.X) in the slab plane).
struct NcLine {
    float c0, ck, cs;
};
__device__ __forceinline__ NcLine nc_line(const CtView &V, const SlabCoef &c, float F) {
    const float tu = F - V.Cu;
    const float rPl = -1.f / fmaf(V.Ku, c.ul, -tu * c.nl);
    return NcLine{fmaf(V.Ku, c.u3, -tu * c.n3) * rPl, fmaf(V.Ku, c.uk, -tu * c.nk) * rPl,
                  fmaf(V.Ku, c.us, -tu * c.ns) * rPl};
}

constexpr int kNcMaxV = 1024;  // voxels cached per round
constexpr int kNcViewBlock = 32;  // views of one tile adjacent in the grid

template <int NA> struct NcCache {
    float4 Fv[2][kNcMaxV];  // rows 4 g0 .. 4 g0 + 7 of the tile
    float Fu[NA][kNcMaxV];
    int2 ag[kNcMaxV];       // (a0, g0)
};

// Forward: CTA = 64 cells x 64 rows of one view, 256 threads; thread (tx, ty)
// owns cells A0 + 4 tx .. + 3 and rows B0 + 4 ty .. + 3 (16 sums).
template <typename TIn, int KIND, int NA, int NB>
__global__ void __launch_bounds__(256, 3)
nc_fwd(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol, const TIn *__restrict__ volZ,
       void *__restrict__ sino, int out_t, int tiles_u, int tiles_v) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    NcCache<NA> &S = *reinterpret_cast<NcCache<NA> *>(smem_raw);
    __shared__ NcBox tile;  // the CTA's box coefficients (read as broadcasts)
    // CTA order: kNcViewBlock consecutive views of one tile, then tiles, then
    // view blocks.  Neighbouring views of a tile read nearly the same voxels,
    // so CTAs resident together share their slabs in L2.
    int bx = blockIdx.x;
    const int vl = bx % kNcViewBlock; bx /= kNcViewBlock;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int tv = bx % tiles_v; bx /= tiles_v;
    const int nvb = (g.nview + kNcViewBlock - 1) / kNcViewBlock;
    const int v = (bx % nvb) * kNcViewBlock + vl;
    const int bt = bx / nvb;
    if (v >= g.nview) return;  // the last block's missing views (whole CTA)
    const int tid = threadIdx.y * 16 + threadIdx.x;
    const int A0 = tu * 64, B0 = tv * 64;
    const int a = A0 + 4 * threadIdx.x, ty = threadIdx.y, rb = B0 + 4 * ty;
    const CtView &V = views[v];
    if (V.nc_tile) return;  // the tile sums' (whole CTA)
    const int main_y = V.main_y;
    const SlabCoef sc = slab_coef(V, main_y);
    const float mu = (KIND == NC_DD ? V.m_dd_u : V.m_sf_u) + 0.5f + kSearchPad;
    const float mv = (KIND == NC_TT ? V.m_tt_v : V.m_sf_v) + 0.5f + kSearchPad;
    const int nslab = main_y ? g.ny : g.nx, nlat = main_y ? g.nx : g.ny;
    const size_t nvox = (size_t)g.nx * g.ny * g.nz;
    const TIn *x = vol + (size_t)bt * nvox;
    const TIn *xz = volZ ? volZ + (size_t)bt * nvox : nullptr;
    if (tid == 0) tile = nc_box_coef(V, sc, A0 - mu, A0 + 63.f + mu, B0 - mv, B0 + 63.f + mv);
    const NcBox cell = nc_box_coef(V, sc, a - mu, a + 3.f + mu, rb - mv, rb + 3.f + mv);
    // the thread's u window per row k: between two lines of constant fu
    const NcLine ln1 = nc_line(V, sc, a - mu), ln2 = nc_line(V, sc, a + 3.f + mu);
    const bool lines = isfinite(ln1.c0) && isfinite(ln1.ck) && isfinite(ln1.cs) && isfinite(ln2.c0) &&
                       isfinite(ln2.ck) && isfinite(ln2.cs);
    const bool live = a < g.nu && rb < g.nv;
    // sums of rows rb + r, cells (a, a + 1) and (a + 2, a + 3): packed FP32x2
    float2 acc[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) acc[r][c] = make_float2(0.f, 0.f);
    __syncthreads();
    for (int s = 0; s < nslab; ++s) {
        const float fs = (float)s;
        int L0, L1, K0, K1;
        if (!nc_box(tile, fs, nlat, g.nz, L0, L1, K0, K1)) continue;  // uniform over the CTA
        int l0 = 0, l1 = -1, k0 = 0, k1 = -1;
        const bool mine = live && nc_box(cell, fs, nlat, g.nz, l0, l1, k0, k1);
        // rounds of nl x nk voxels, k fastest (contiguous in the z-major copy)
        const int nk = min(K1 - K0 + 1, kNcMaxV);
        const int nlr = kNcMaxV / nk;
        for (int kc = K0; kc <= K1; kc += nk) {
            const int nkr = min(nk, K1 - kc + 1);
            for (int lc = L0; lc <= L1; lc += nlr) {
                const int nl = min(nlr, L1 - lc + 1);
                __syncthreads();
                for (int idx = tid; idx < nl * nkr; idx += 256) {
                    const int l = lc + idx / nkr, k = kc + idx % nkr;
                    const int i = main_y ? l : s, j = main_y ? s : l;
                    NcFp<NA, NB> P;
                    nc_fp<KIND, NA, NB>(V, g, nc_col<KIND>(V, g, i, j), (float)k, P);
                    const float xv = xz ? ld(xz, ((size_t)j * g.nx + i) * g.nz + k)
                                        : ld(x, ((size_t)k * g.ny + j) * g.nx + i);
                    const float w = P.amp * xv;
#pragma unroll
                    for (int q = 0; q < NA; ++q) S.Fu[q][idx] = P.Fu[q] * w;
                    // first 4-row group of the footprint and its offset in it
                    const int rel = P.b0 - B0;
                    const int g0 = rel >= 0 ? rel >> 2 : -((3 - rel) >> 2);
                    const int o = rel - 4 * g0;  // 0 .. 3
                    float w8[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t) w8[t] = 0.f;
#pragma unroll
                    for (int oo = 0; oo < 4; ++oo)
                        if (o == oo) {
#pragma unroll
                            for (int q = 0; q < NB; ++q) w8[oo + q] = P.Fv[q];
                        }
                    S.Fv[0][idx] = make_float4(w8[0], w8[1], w8[2], w8[3]);
                    S.Fv[1][idx] = make_float4(w8[4], w8[5], w8[6], w8[7]);
                    S.ag[idx] = make_int2(P.a0, g0);
                }
                __syncthreads();
                if (!mine) continue;
                const int la = max(l0, lc), lb = min(l1, lc + nl - 1);
                const int ka = max(k0, kc), kb = min(k1, kc + nkr - 1);
                const float ls1 = fmaf(ln1.cs, fs, ln1.c0), ls2 = fmaf(ln2.cs, fs, ln2.c0);
                for (int k = ka; k <= kb; ++k) {
                    int lo = la, hi = lb;
                    if (lines) {  // lateral range of row k (1e-3 voxel rounding guard)
                        const float fk = (float)k;
                        const float u1 = fmaf(ln1.ck, fk, ls1), u2 = fmaf(ln2.ck, fk, ls2);
                        lo = max(la, (int)ceilf(fminf(u1, u2) - 1e-3f));
                        hi = min(lb, (int)floorf(fmaxf(u1, u2) + 1e-3f));
                    }
                    int idx = (lo - lc) * nkr + (k - kc);
                    for (int l = lo; l <= hi; ++l, idx += nkr) {
                        const int2 ag = S.ag[idx];
                        const int d = a - ag.x;  // first cell of the thread in the footprint
                        const int gd = ty - ag.y;
                        if ((unsigned)gd > 1u || (unsigned)(d + 3) >= (unsigned)(NA + 3)) continue;  // -4 < d < NA
                        const float4 fv = S.Fv[gd][idx];
                        // Fu[d + c][idx] for the thread's cells c: one base offset
                        const float *fu = &S.Fu[0][0];
                        const int off = d * kNcMaxV + idx;
                        float wu[4];
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            wu[c] = (unsigned)(d + c) < (unsigned)NA ? fu[off + c * kNcMaxV] : 0.f;
                        const float2 w01 = make_float2(wu[0], wu[1]), w23 = make_float2(wu[2], wu[3]);
                        const float fr[4] = {fv.x, fv.y, fv.z, fv.w};
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float2 f = make_float2(fr[r], fr[r]);
                            acc[r][0] = __ffma2_rn(w01, f, acc[r][0]);
                            acc[r][1] = __ffma2_rn(w23, f, acc[r][1]);
                        }
                    }
                }
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int b = rb + r;
        if (b >= g.nv) break;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int ac = a + c;
            const float2 p = acc[r][c >> 1];
            const float sum = (c & 1) ? p.y : p.x;
            if (ac < g.nu)
                st_out(g, sino, (((size_t)bt * g.nview + v) * g.nv + b) * g.nu + ac,
                       KIND != NC_SF ? sum * nc_cell_factor<KIND>(V, g, ac, b) : sum, out_t);
        }
    }
}

// ------------------------------------------------------------ forward (tile sums)
// CTA = a tile of 32 cells x R rows of one view; each of its four warps sums
// every fourth slab into a copy of the tile of its own in shared memory (with a
// margin as wide as a footprint, so that adds need no bounds test), and the
// copies are added at the end.  A warp runs over the columns of a slab that can
// reach the tile, four columns a quarter of the slab apart at a time, eight
// consecutive voxels of each; a lane evaluates its voxel's footprint once and
// adds its weights.  Lanes add row by row of their footprints with the warp in
// step.  Consecutive voxels of a column start at different rows when an axial
// footprint is at least a row high, so no two lanes of a column touch a cell in
// the same step; where a height between half a row and one lets neighbours share
// a row, or the four columns' cells are not apart, the lanes take turns (decided
// by votes on the footprints themselves).  The order of every sum is fixed, and
// nothing that orders it depends on another view: which views are summed so is
// decided view by view (CtView::nc_tile; the others take the gather above), and who
// votes on sharing rows does not depend on the margins, which follow the scan's NA
// and NB.
//
// Why two lanes never add to one cell in the same step.  The cells a column adds
// to over its eight voxels lie between a0 and a0 + 3 (NA - 1) of its footprints.
// Each transaxial corner moves one way along u with k, so the lowest a0 is that of
// the first or the last voxel, up to one cell of rounding.  The highest may exceed
// both, where corners move opposite ways, by no more than the corners' offsets from
// the centre change, since the centre itself moves one way: less than a cell by the
// host's condition on nc_tile.  So ranges taken from the end voxels that are more
// than two cells apart do not meet; and as centres are monotone along the slab,
// neighbouring groups that are apart leave all four apart.
//
// Against the gather above it evaluates the same footprints (1.2 per update)
// but adds each weight once, where a gathering thread visits every voxel that
// might reach its cells (five visits of 16 products per update for about eight
// non-zero weights).  192^3 / 250 views / 384^2 FP16 SF-TR: gather 52.8 ms, tile
// sums 27.4 ms (bound by instruction issue and L1); 64^3 / 90 views DD 924 -> 390 us.
template <int NA, int NB> struct ScTile {
    static constexpr int kMc = NA - 1, kMr = NB - 1;  // margins
    static constexpr int kPitch = (32 + 2 * kMc) | 1;
    static constexpr int floats(int R) { return (R + 2 * kMr) * kPitch; }
};
constexpr int kScWarps = 4;

template <typename TIn, int KIND, int NA, int NB>
__global__ void __launch_bounds__(32 * kScWarps, 6)
nc_fwd_tile(CtGrid g, const CtView *__restrict__ views, const TIn *__restrict__ vol, bool zmajor, void *__restrict__ sino,
            int out_t, int tiles_u, int tiles_v, int R) {
    using Tile = ScTile<NA, NB>;
    constexpr int P_ = Tile::kPitch;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ CtView V;
    __shared__ NcBox box;
    const int lane = threadIdx.x, w = threadIdx.y;
    float *tile = reinterpret_cast<float *>(smem_raw) + w * Tile::floats(R);
    // CTA order: as in nc_fwd, kNcViewBlock views of one tile adjacent
    int bx = blockIdx.x;
    const int vl = bx % kNcViewBlock; bx /= kNcViewBlock;
    const int tu = bx % tiles_u; bx /= tiles_u;
    const int tv = bx % tiles_v; bx /= tiles_v;
    const int nvb = (g.nview + kNcViewBlock - 1) / kNcViewBlock;
    const int v = (bx % nvb) * kNcViewBlock + vl;
    const int bt = bx / nvb;
    if (v >= g.nview) return;  // the last block's missing views (whole CTA)
    const int A0 = tu * 32, B0 = tv * R;
    if (w == 0) {
        if (lane < (int)(sizeof(CtView) / sizeof(float4)))
            reinterpret_cast<float4 *>(&V)[lane] = __ldg(reinterpret_cast<const float4 *>(views + v) + lane);
        __syncwarp();
        if (lane == 0) {
            const float mu = (KIND == NC_DD ? V.m_dd_u : V.m_sf_u) + 0.5f + kSearchPad;
            const float mv = (KIND == NC_TT ? V.m_tt_v : V.m_sf_v) + 0.5f + kSearchPad;
            const int Bl = min(B0 + R, g.nv) - 1, Al = min(A0 + 32, g.nu) - 1;
            box = nc_box_coef(V, slab_coef(V, V.main_y), A0 - mu, Al + mu, B0 - mv, Bl + mv);
        }
    }
    for (int q = lane; q < Tile::floats(R); q += 32) tile[q] = 0.f;
    __syncthreads();
    if (!V.nc_tile) return;  // the gather's (whole CTA)
    const int main_y = V.main_y;
    const SlabCoef sc = slab_coef(V, main_y);
    const int nslab = main_y ? g.ny : g.nx, nlat = main_y ? g.nx : g.ny;
    const float hl = main_y ? g.dx : g.dy, hs = main_y ? g.dy : g.dx;
    const float ol = main_y ? V.o[0] : V.o[1], os = main_y ? V.o[1] : V.o[0];
    // strides along z, the lateral axis and the slabs: of the z-major copy, or of the
    // volume itself where the copy could not be had
    const size_t pk = zmajor ? 1 : (size_t)g.nx * g.ny, pc = zmajor ? g.nz : 1;
    const size_t pl = pc * (main_y ? 1 : g.nx), ps = pc * (main_y ? g.nx : 1);
    const TIn *xz = vol + (size_t)bt * g.nx * g.ny * g.nz;
    const int grp = lane >> 3;
    for (int s = w; s < nslab; s += kScWarps) {
        int L0, L1, K0, K1;
        const float fs = (float)s;
        if (!nc_box(box, fs, nlat, g.nz, L0, L1, K0, K1)) continue;  // uniform over the warp
        const int nq = (L1 - L0 + 4) >> 2;
        const float ws = fmaf(fs, hs, os), wsa = fabsf(ws), ws2 = ws * ws;
        const int l0 = L0 + grp * nq;
        for (int kc = K0; kc <= K1; kc += 8) {
            const int k = kc + (lane & 7);
            const float fk = (float)k;
            const TIn *xk = xz + s * ps + l0 * pl + k * pk;
            for (int t = 0; t < nq; ++t, xk += pl) {
                const bool in = k <= K1 && l0 + t <= L1;
                const float xv = in ? ld(xk, 0) : 0.f;
                const float fl = (float)(l0 + t);
                NcCol C;
                C.cu = fmaf(sc.ul, fl, fmaf(sc.us, fs, sc.u3));
                C.cn = fmaf(sc.nl, fl, fmaf(sc.ns, fs, sc.n3));
                C.cv = fmaf(sc.vl, fl, fmaf(sc.vs, fs, sc.v3));
                if (KIND == NC_SF) {
                    const float wl = fmaf(fl, hl, ol);
                    C.r2 = fmaf(wl, wl, ws2);
                    C.im = __fdividef(g.dx, fmaxf(fabsf(wl), wsa));
                }
                NcFp<NA, NB> P;
                nc_fp<KIND, NA, NB>(V, g, C, fk, P);
                const int c0 = P.a0 - A0 + Tile::kMc, r0 = P.b0 - B0 + Tile::kMr;
                const bool hit = in && (unsigned)c0 < 32u + Tile::kMc && (unsigned)r0 < (unsigned)(R + Tile::kMr);
                if (!__any_sync(~0u, hit)) continue;
                // lanes that may touch a cell in the same step take turns
                // (every lane takes part in the exchanges; a column's first
                // cell is monotone in k, and in l at a given k)
                const int below = __shfl_up_sync(~0u, P.b0, 1, 8);
                const int af = __shfl_sync(~0u, P.a0, 0, 8), al = __shfl_sync(~0u, P.a0, min(7, K1 - kc), 8);
                const bool wide = __any_sync(~0u, hit && P.n > 4);
                const int mn = min(af, al), mx = max(af, al) + (wide ? NA : min(NA, 4)) - 1;  // cells added to
                const int nmn = __shfl_down_sync(~0u, mn, 8), nmx = __shfl_down_sync(~0u, mx, 8);
                const bool odd = __any_sync(~0u, in && (lane & 7) && below == P.b0);
                const bool near = __any_sync(~0u, lane < 24 && !(nmn > mx + 2 || mn > nmx + 2));
                const int nph = (odd ? 2 : 1) * (near ? 4 : 1);
                const int mine = (odd ? lane & 1 : 0) + (near ? (odd ? 2 : 1) * grp : 0);
                const float val = P.amp * xv;
#pragma unroll
                for (int c = 0; c < NA; ++c) P.Fu[c] *= val;
                float *t0 = tile + (hit ? r0 * P_ + c0 : 0);
                for (int ph = 0; ph < nph; ++ph) {
                    const bool go = hit && mine == ph;
#pragma unroll
                    for (int q = 0; q < NB; ++q) {
                        if (go && P.Fv[q] != 0.f) {
#pragma unroll
                            for (int c = 0; c < (NA < 4 ? NA : 4); ++c)
                                t0[q * P_ + c] = fmaf(P.Fu[c], P.Fv[q], t0[q * P_ + c]);
                            if (NA > 4 && wide) {
#pragma unroll
                                for (int c = 4; c < NA; ++c)
                                    t0[q * P_ + c] = fmaf(P.Fu[c], P.Fv[q], t0[q * P_ + c]);
                            }
                        }
                        __syncwarp();
                    }
                }
            }
        }
    }
    __syncthreads();
    const int a = A0 + lane;
    if (a >= g.nu) return;
    const float *t0 = reinterpret_cast<const float *>(smem_raw) + Tile::kMr * P_ + lane + Tile::kMc;
    for (int r = w; r < R && B0 + r < g.nv; r += kScWarps) {
        float sum = t0[r * P_];
#pragma unroll
        for (int q = 1; q < kScWarps; ++q) sum += t0[q * Tile::floats(R) + r * P_];
        st_out(g, sino, (((size_t)bt * g.nview + v) * g.nv + B0 + r) * g.nu + a,
               KIND != NC_SF ? sum * nc_cell_factor<KIND>(V, g, a, B0 + r) : sum, out_t);
    }
}

// Rows of a tile: about four passes of eight voxels at the magnification of about
// 1.5 that cone-beam scanners have.  From the sizes alone, so that a view's
// result does not depend on the other views.
inline int sc_rows(const CtGrid &g) {
    const float r = 42.f * g.dz / g.dv - 2.f;
    return r < 16.f ? 16 : r > 56.f ? 56 : (int)r;
}

namespace {
template <typename TIn, int KIND, int NA, int NB> struct NcFwd {
    static cudaError_t go(const CtGrid &g, const CtView *views, const void *in, void *out, int out_t, int batch,
                          cudaStream_t st) {
        const TIn *src = static_cast<const TIn *>(in);
        cudaError_t e = cudaSuccess;
        // a z-major copy of the volume (pooled workspace) makes each round's
        // reads contiguous along k; without it the reads are strided
        TIn *xZ = nullptr;
        const size_t n = (size_t)g.nx * g.ny * g.nz * batch;
        if (workspace_alloc_copy((void **)&xZ, n * sizeof(TIn), g, st) != cudaSuccess) {
            cudaGetLastError();
            xZ = nullptr;
        } else if ((e = zmajor_copy(sizeof(TIn), src, xZ, g.nx, g.ny, g.nz, g.nz, batch, st)) != cudaSuccess) {
            workspace_free(xZ, st);
            return e;
        }
        const size_t nvb = (g.nview + kNcViewBlock - 1) / kNcViewBlock;
        if (g.nc_tile) {  // the views that allow tile sums
            const int R = sc_rows(g);
            const int tiles_c = (g.nu + 31) / 32, tiles_r = (g.nv + R - 1) / R;
            const size_t sm = sizeof(float) * kScWarps * (size_t)ScTile<NA, NB>::floats(R);
            e = cudaFuncSetAttribute(nc_fwd_tile<TIn, KIND, NA, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
            if (e == cudaSuccess) {
                const dim3 grd((unsigned)((size_t)kNcViewBlock * tiles_c * tiles_r * nvb * batch));
                nc_fwd_tile<TIn, KIND, NA, NB><<<grd, dim3(32, kScWarps), sm, st>>>(g, views, xZ ? xZ : src, xZ != nullptr, out,
                                                                                   out_t, tiles_c, tiles_r, R);
                e = cudaGetLastError();
            }
        }
        if (e == cudaSuccess && g.nc_gather) {  // the others
            const size_t smem = sizeof(NcCache<NA>);
            e = cudaFuncSetAttribute(nc_fwd<TIn, KIND, NA, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e == cudaSuccess) {
                const int tiles_u = (g.nu + 63) / 64, tiles_v = (g.nv + 63) / 64;
                dim3 blk(16, 16), grd((unsigned)((size_t)kNcViewBlock * tiles_u * tiles_v * nvb * batch));
                nc_fwd<TIn, KIND, NA, NB><<<grd, blk, smem, st>>>(g, views, src, xZ, out, out_t, tiles_u, tiles_v);
                e = cudaGetLastError();
            }
        }
        const cudaError_t ef = workspace_free(xZ, st);
        return e != cudaSuccess ? e : ef;
    }
};
}  // namespace

cudaError_t launch_nc_fwd(int kind, const CtGrid &g, const CtView *views, int in_t, const void *in, int out_t,
                          void *out, int batch, cudaStream_t st) {
    return nc_dispatch<NcFwd>(kind, in_t, g, views, in, out, out_t, batch, st);
}

}  // namespace ctp
