// k_ray.cuh -- what the ray-driven kernels of fan-beam and cone-beam geometry
// share: the ray of a cell, and a run of its chords (Siddon 1985).
#pragma once
#include "ct_device.cuh"

namespace ctp {

// world direction from the source to the centre of cell (a, b)
template <bool CURVED>
__device__ __forceinline__ void ray_dir(const CtView &V, const CtGrid &g, int a, int b, float d[3]) {
    const float Vb = g.dv * ((float)b - V.Cv);
    float cn_, cu_;
    if (CURVED) {
        float sg, cg;
        sincosf(((float)a - V.Cu) / V.Ku, &sg, &cg);
        cn_ = V.D * cg;
        cu_ = V.D * sg;
    } else {
        cn_ = V.D;
        cu_ = g.du * ((float)a - V.Cu);
    }
#pragma unroll
    for (int m = 0; m < 3; ++m) d[m] = fmaf(cn_, V.nn[m], fmaf(cu_, V.eu[m], Vb * V.ev[m]));
}

// Sums of chord x value over the runs grp, grp + 1, .. (N of them) of NG runs of slabs
// of the ray of cell (a, b); the caller adds the runs and multiplies by the ray's
// length `len`.  (A run's sum is the same whichever thread forms it.)
// TWO: fan beam, the ray stays in the one slice.
//
// The chord lengths are Siddon's, taken slab by slab along the axis on which the
// ray moves most (in voxels): inside a slab either other index changes by at
// most one, so a slab meets at most three voxels, split where the ray crosses
// into the next lateral and the next axial index.  Every crossing's parameter
// (from the entry point) is formed from its plane alone, so runs of slabs are
// independent, no load waits for the one before, and neighbouring rays stay in
// the same slab, so their loads coalesce.  Axes along which the ray descends are
// mirrored (indices and strides negated).  volT (may be null): a copy of the
// volume whose fastest axis is y, for rays along x.
template <typename TIn, bool CURVED, bool TWO, int NG, int N>
__device__ __forceinline__ void ray_runs(const CtView &V, const CtGrid &g, int a, int b, const TIn *__restrict__ vol,
                                         const TIn *__restrict__ volT, int grp, float &len, float (&sum)[N]) {
    constexpr int NAX = TWO ? 2 : 3;
    float d[3];
    ray_dir<CURVED>(V, g, a, b, d);
    len = sqrtf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])));
    const float h[3] = {g.dx, g.dy, g.dz};
    const int n[3] = {g.nx, g.ny, g.nz};
    // source and direction in voxel-index units; voxel i spans [i - 1/2, i + 1/2)
    float S[3], D[3], tin = 0.f, tout = 1.f;
    bool hit = true;
#pragma unroll
    for (int m = 0; m < NAX; ++m) {
        S[m] = -V.o[m] / h[m];
        D[m] = d[m] / h[m];
        const float lo = -0.5f, hi = (float)n[m] - 0.5f;
        if (D[m] == 0.f) {
            if (!(S[m] >= lo && S[m] < hi)) hit = false;
        } else {
            const float t1 = (lo - S[m]) / D[m], t2 = (hi - S[m]) / D[m];
            tin = fmaxf(tin, fminf(t1, t2));
            tout = fminf(tout, fmaxf(t1, t2));
        }
    }
#pragma unroll
    for (int q = 0; q < N; ++q) sum[q] = 0.f;
    if (!(hit && tout > tin)) return;
    const float T = tout - tin;
    // mirrored axes: entry point, speed, crossing-parameter step, index range
    float q[3], inv[3], lo[3], hi[3];
    ptrdiff_t st[3] = {1, (ptrdiff_t)g.nx, (ptrdiff_t)g.nx * g.ny};
    const bool z = !TWO && fabsf(D[2]) > fabsf(D[0]) && fabsf(D[2]) > fabsf(D[1]);
    const bool y = !z && fabsf(D[1]) >= fabsf(D[0]);
    const bool swap = !y && !z && volT != nullptr;
    if (swap) {
        st[0] = g.ny;
        st[1] = 1;
    }
#pragma unroll
    for (int m = 0; m < NAX; ++m) {
        const float e = fmaf(tin, D[m], S[m]);
        const bool neg = D[m] < 0.f;
        q[m] = neg ? -e : e;
        D[m] = fabsf(D[m]);
        inv[m] = D[m] != 0.f ? 1.f / D[m] : 0.f;
        lo[m] = neg ? 1.f - (float)n[m] : 0.f;
        hi[m] = neg ? 0.f : (float)(n[m] - 1);
        if (neg) st[m] = -st[m];
    }
    // main axis m and the others p, r
    auto pick = [&](const float *v, int w) {  // w: 0 main, 1 lateral, 2 the remaining axis
        if (TWO) return w == 0 ? (y ? v[1] : v[0]) : (y ? v[0] : v[1]);
        return w == 0 ? (z ? v[2] : y ? v[1] : v[0]) : w == 1 ? (y || z ? v[0] : v[1]) : (z ? v[1] : v[2]);
    };
    const ptrdiff_t tm = z ? st[2] : y ? st[1] : st[0], tp = y || z ? st[0] : st[1], tr = z ? st[1] : st[2];
    auto index = [](float x, float l, float u) { return fminf(fmaxf(floorf(x + 0.5f), l), u); };
    const float Dm = pick(D, 0), qm = pick(q, 0), im = pick(inv, 0), um = pick(hi, 0);
    const float c0 = index(qm, pick(lo, 0), um);  // entry slab
    // slabs to the volume's end, or to the ray's
    const int nsl = (int)fminf(um - c0 + 1.f, floorf(T * Dm) + 3.f), per = (nsl + NG - 1) / NG;
    constexpr float kNever = 3.0e38f;
#pragma unroll 1
    for (int run = 0; run < N; ++run) {
        const int i0 = (grp + run) * per, i1 = min(i0 + per, nsl);
        if (i0 >= i1) return;
        float cm = c0 + (float)i0;  // the slab's index
        float ta = i0 == 0 ? 0.f : fminf(fmaxf((cm - 0.5f - qm) * im, 0.f), T);
        // lateral index, and the parameter at which the next one begins
        const float qp = pick(q, 1), ip = pick(inv, 1), up = pick(hi, 1);
        float jp = index(fmaf(ta, pick(D, 1), qp), pick(lo, 1), up);
        float np = ip != 0.f && jp < up ? (jp + 0.5f - qp) * ip : kNever;
        ptrdiff_t off = (ptrdiff_t)cm * tm + (ptrdiff_t)jp * tp;
        float qr = 0.f, ir = 0.f, ur = 0.f, jr = 0.f, nr = kNever;
        if (!TWO) {
            qr = pick(q, 2); ir = pick(inv, 2); ur = pick(hi, 2);
            jr = index(fmaf(ta, pick(D, 2), qr), pick(lo, 2), ur);
            nr = ir != 0.f && jr < ur ? (jr + 0.5f - qr) * ir : kNever;
            off += (ptrdiff_t)jr * tr;
        }
        const TIn *x = (swap ? volT : vol) + off;
        float acc = 0.f;
        for (int i = i0; i < i1 && ta < T; ++i, x += tm, cm += 1.f) {
            const float te = fminf(fmaxf((cm + 0.5f - qm) * im, ta), T);
            const bool xp = np < te, xr = !TWO && nr < te;
            const float cp = xp ? fmaxf(np, ta) : te, cr = xr ? fmaxf(nr, ta) : te;
            const float e1 = TWO ? cp : fminf(cp, cr);
            acc = fmaf(e1 - ta, ld(x, 0), acc);
            if (TWO) {
                if (xp) {
                    x += tp;
                    acc = fmaf(te - cp, ld(x, 0), acc);
                    jp += 1.f;
                    np = jp < up ? (jp + 0.5f - qp) * ip : kNever;
                }
            } else if (xp || xr) {
                const float e2 = fmaxf(cp, cr);
                acc = fmaf(e2 - e1, ld(x + (xp && (!xr || cp < cr) ? tp : tr), 0), acc);
                if (xp) {
                    x += tp;
                    jp += 1.f;
                    np = jp < up ? (jp + 0.5f - qp) * ip : kNever;
                }
                if (xr) {
                    x += tr;
                    jr += 1.f;
                    nr = jr < ur ? (jr + 0.5f - qr) * ir : kNever;
                }
                if (xp && xr) acc = fmaf(te - e2, ld(x, 0), acc);
            }
            ta = te;
        }
        // (registers, for any N)
#pragma unroll
        for (int q = 0; q < N; ++q) sum[q] = q == run ? acc : sum[q];
    }
}

}  // namespace ctp
