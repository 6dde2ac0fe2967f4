// lbm_device.cuh -- device-side building blocks shared by the step, density and
// measurement kernels: column coordinates with periodic wrap, and the pull of
// one cell's 2 x 19 populations with half-way bounce-back (Eq. 1, left-hand side).
#pragma once

#include "lbm_internal.h"

namespace lbmk {

// Wrap a coordinate one step beyond the box; ok is cleared when it falls beyond
// a closed edge (the returned value is then clamped and must not be used).
__device__ __forceinline__ int wrap1(int v, int n, int periodic, bool& ok) {
    if (v < 0) {
        if (periodic) return v + n;
        ok = false;
        return 0;
    }
    if (v >= n) {
        if (periodic) return v - n;
        ok = false;
        return n - 1;
    }
    return v;
}

// Neighbour coordinate for a source lookup: wrapped, or clamped into the box
// (a clamped value is only ever used behind a bounce-back bit).
__device__ __forceinline__ int nb1(int v, int n, int periodic) {
    if (v < 0) return periodic ? v + n : 0;
    if (v >= n) return periodic ? v - n : n - 1;
    return v;
}

// The x/y part of a cell's pull addresses.  xo[i] / yo[i] are the (wrapped)
// x offset and y row offset of x - 1 + i / y - 1 + i.
struct Column {
    int xo[3];
    int yo[3];
    bool ok;  // the column exists (inside the box or a periodic image)
};

__device__ __forceinline__ Column make_column(int gx, int gy, const Geom& g) {
    Column c;
    c.ok = true;
    int x = wrap1(gx, g.nx, g.px, c.ok);
    int y = wrap1(gy, g.ny, g.py, c.ok);
    c.xo[0] = nb1(x - 1, g.nx, g.px);
    c.xo[1] = x;
    c.xo[2] = nb1(x + 1, g.nx, g.px);
    c.yo[0] = nb1(y - 1, g.ny, g.py) * g.nx;
    c.yo[1] = y * g.nx;
    c.yo[2] = nb1(y + 1, g.ny, g.py) * g.nx;
    return c;
}

// Pull the populations of one cell whose geometry word w is known:
//   f_k(x) = f*_k(x - e_k)   if x - e_k is fluid for the component,
//   f_k(x) = f*_kbar(x)      otherwise (half-way bounce-back),
// from the post-collision array fin[(s*19 + k) * plane + cell].  zz is the
// cell's (wrapped) plane.  Returns the component densities (0 where a component
// is not fluid): with ILP in four interleaved partial sums, otherwise in k order.
// With KEEP the pulled values are left in f.
template <bool KEEP, bool ILP = false>
__device__ __forceinline__ void pull_known(const float* __restrict__ fin, const uint32_t* __restrict__ nbr_nw,
                                           const Geom& g, const Column& c, int zz, int cell, uint32_t w,
                                           float (&f)[2][Q], float& rw, float& rn) {
    rw = 0.f;
    rn = 0.f;
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID || cls == CLS_OUTSIDE) return;
    // away from periodic seams the source of direction k is cell - (ex + ey nx + ez nxy)
    const bool seam = (g.px && (c.xo[1] == 0 || c.xo[1] == g.nx - 1)) ||
                      (g.py && (c.yo[1] == 0 || c.yo[1] == (g.ny - 1) * g.nx)) ||
                      (g.pz && (zz == 0 || zz == g.nz - 1));
    int zo[3];
    zo[0] = nb1(zz - 1, g.nz, g.pz) * g.nxy;
    zo[1] = zz * g.nxy;
    zo[2] = nb1(zz + 1, g.nz, g.pz) * g.nxy;
    const uint32_t wn = (cls == CLS_MEMBRANE) ? 0u : ((w & BIT_NW_DIFF) ? __ldg(nbr_nw + cell) : w);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (s == 1 && cls == CLS_MEMBRANE) {
            if (KEEP) {
#pragma unroll
                for (int k = 0; k < Q; ++k) f[1][k] = 0.f;
            }
            break;
        }
        const uint32_t bits = s == 0 ? w : wn;
        const float* fs = fin + (size_t)s * Q * g.plane;
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            int src;
            if (!seam) src = cell - (EX(k) + EY(k) * g.nx + EZ(k) * g.nxy);
            else src = zo[1 - EZ(k)] + c.yo[1 - EY(k)] + c.xo[1 - EX(k)];
            const int idx = ((bits >> k) & 1u) ? (OPP(k) * g.plane + cell) : (k * g.plane + src);
            const float v = __ldg(fs + idx);
            if (KEEP) f[s][k] = v;
            if (ILP) a[k & 3] += v;
            else a[0] += v;
        }
        const float r = ILP ? (a[0] + a[1]) + (a[2] + a[3]) : a[0];
        if (s == 0) rw = r;
        else rn = r;
    }
}

// Pull cell (column, z): loads the geometry word, then as pull_known.  Returns
// the word (class CLS_OUTSIDE for a cell beyond a closed edge).
template <bool KEEP>
__device__ __forceinline__ uint32_t pull_cell(const float* __restrict__ fin, const uint32_t* __restrict__ nbr,
                                              const uint32_t* __restrict__ nbr_nw, const Geom& g,
                                              const Column& c, int z, float (&f)[2][Q], float& rw, float& rn,
                                              int& cell_out) {
    rw = 0.f;
    rn = 0.f;
    cell_out = 0;
    bool ok = c.ok;
    const int zz = wrap1(z, g.nz, g.pz, ok);
    if (!ok) return CLS_OUTSIDE << CLS_SHIFT;
    const int cell = zz * g.nxy + c.yo[1] + c.xo[1];
    cell_out = cell;
    const uint32_t w = __ldg(nbr + cell);
    pull_known<KEEP>(fin, nbr_nw, g, c, zz, cell, w, f, rw, rn);
    return w;
}

__device__ __forceinline__ bool fluid_w(uint8_t m) { return !(m & LBM_MASK_SOLID); }
__device__ __forceinline__ bool fluid_nw(uint8_t m) { return !(m & (LBM_MASK_SOLID | LBM_MASK_MEMBRANE)); }

// Geometry words (layout in lbm_internal.h) of cell (x, y, z).  For every
// direction k the pull source x - e_k decides the bounce bit of each component;
// the neighbour x + e_k contributes 36 w_k e_k to the adhesion vector when it is
// grain.
__device__ __forceinline__ void geometry_cell(const uint8_t* __restrict__ mask, uint32_t* __restrict__ nbr,
                                              uint32_t* __restrict__ nbr_nw, uint32_t* __restrict__ adh,
                                              const Geom& g, int x, int y, int z) {
    const long long c = (long long)z * g.nxy + (long long)y * g.nx + x;
    const uint8_t m = __ldg(mask + c);
    uint32_t cls;
    if (m & LBM_MASK_SOLID) cls = CLS_SOLID;
    else if (m & LBM_MASK_INLET) cls = CLS_INLET;
    else if (m & LBM_MASK_OUTLET) cls = CLS_OUTLET;
    else if (m & LBM_MASK_MEMBRANE) cls = CLS_MEMBRANE;
    else cls = CLS_FLUID;
    uint32_t bw = 0, bn = 0;
    int ax = 0, ay = 0, az = 0;
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        bool ok = true;
        const int sx = wrap1(x - EX(k), g.nx, g.px, ok);
        const int sy = wrap1(y - EY(k), g.ny, g.py, ok);
        const int sz = wrap1(z - EZ(k), g.nz, g.pz, ok);
        if (!ok) {
            bw |= 1u << k;
            bn |= 1u << k;
        } else {
            const uint8_t ms = __ldg(mask + (long long)sz * g.nxy + (long long)sy * g.nx + sx);
            if (!fluid_w(ms)) bw |= 1u << k;
            if (!fluid_nw(ms)) bn |= 1u << k;
        }
        bool ok2 = true;
        const int tx = wrap1(x + EX(k), g.nx, g.px, ok2);
        const int ty = wrap1(y + EY(k), g.ny, g.py, ok2);
        const int tz = wrap1(z + EZ(k), g.nz, g.pz, ok2);
        if (ok2) {
            const uint8_t mt = __ldg(mask + (long long)tz * g.nxy + (long long)ty * g.nx + tx);
            if ((mt & LBM_MASK_SOLID) && (mt & LBM_MASK_ADHESIVE)) {
                ax += W36(k) * EX(k);
                ay += W36(k) * EY(k);
                az += W36(k) * EZ(k);
            }
        }
    }
    uint32_t word = bw | (cls << CLS_SHIFT);
    if (bn != bw) word |= BIT_NW_DIFF;
    if (ax || ay || az) word |= BIT_ADH;
    nbr[c] = word;
    nbr_nw[c] = bn;
    adh[c] = (uint32_t)(uint8_t)(int8_t)ax | ((uint32_t)(uint8_t)(int8_t)ay << 8) |
             ((uint32_t)(uint8_t)(int8_t)az << 16);
}

// A thread's measurement sums (definitions in lbm.h).  GB300 has little FP64
// throughput, and a division there is some twenty FP64 instructions: the sums
// that need 64 bits (masses and Eq. 5 pressures) take eight FP64 instructions a
// cell, the counts are integers, and the phase of a cell is decided in FP32 where
// that is exact or far from the threshold (192^3 sample, push layout: 0.72 ->
// 0.21 ms; 0.12 ms is its HBM floor).
struct MeasureSums {
    double mass[2] = {0.0, 0.0};
    double p[4] = {0.0, 0.0, 0.0, 0.0};  // 3 x Eq. 5: bulk wetting, bulk non-wetting, inlet, outlet
    unsigned n[9] = {};                  // MS_N_FLUID .. MS_N_NEGATIVE

    __device__ __forceinline__ void count(int i, bool yes) { n[i - MS_N_FLUID] += yes ? 1u : 0u; }

    __device__ __forceinline__ void add(uint32_t cls, float rw, float rn, double G) {
        if (cls == CLS_SOLID || cls == CLS_OUTSIDE) return;
        const bool has_nw = cls != CLS_MEMBRANE;
        const double dw = rw, dn = rn;
        mass[0] += dw;
        if (has_nw) mass[1] += dn;
        const bool fw = isfinite(rw), fn = isfinite(rn);
        count(MS_N_NONFINITE, !fw);
        count(MS_N_NONFINITE, has_nw && !fn);
        count(MS_N_NEGATIVE, fw && rw < 0.f);
        count(MS_N_NEGATIVE, has_nw && fn && rn < 0.f);
        if (!has_nw) return;
        const double p3 = fma(G * dw, dn, dw + dn);
        if (cls == CLS_INLET) { p[2] += p3; count(MS_N_IN, true); return; }
        if (cls == CLS_OUTLET) { p[3] += p3; count(MS_N_OUT, true); return; }
        count(MS_N_FLUID, true);
        count(MS_N_W, rw > rn);
        // phi = (rw - rn) / (rw + rn): for a positive sum |phi| < 0.5 is rw < 3 rn and
        // rn < 3 rw, and the sign of a fused multiply-add is exact; phi > 0.9 is
        // rw > 19 rn, decided in FP32 unless the two are within 1e-4 of each other
        const float y = rw + rn, a = fmaf(-19.f, rn, rw), b = fmaf(-19.f, rw, rn), near = 1e-4f * y;
        if (y > 0.f && y < 1e30f && fabsf(a) > near && fabsf(b) > near) {
            count(MS_N_INTERFACE, fmaf(3.f, rn, -rw) > 0.f && fmaf(3.f, rw, -rn) > 0.f);
            count(MS_N_BULK_W, a > 0.f);
            count(MS_N_BULK_NW, b > 0.f);
            if (a > 0.f) p[0] += p3;
            if (b > 0.f) p[1] += p3;
        } else {
            const double phi = (dw - dn) / (dw + dn);
            count(MS_N_INTERFACE, fabs(phi) < 0.5);
            if (phi > 0.9) { p[0] += p3; count(MS_N_BULK_W, true); }
            if (phi < -0.9) { p[1] += p3; count(MS_N_BULK_NW, true); }
        }
    }

    // The sums of a block of WARPS warps into out[NMEAS] (all threads call it).
    template <int WARPS>
    __device__ __forceinline__ void store(double* __restrict__ out) const {
        __shared__ double red[WARPS][NMEAS];
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
        const double d[6] = {mass[0], mass[1], p[0], p[1], p[2], p[3]};
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            double v = d[i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) red[wid][i] = i < 2 ? v : v * (1.0 / 3.0);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const unsigned v = __reduce_add_sync(0xffffffffu, n[i]);
            if (lane == 0) red[wid][MS_N_FLUID + i] = (double)v;
        }
        if (lane == 0) red[wid][MS_SPARE] = 0.0;
        __syncthreads();
        if (tid < NMEAS) {
            double v = 0.0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) v += red[w][tid];
            out[tid] = v;
        }
    }
};

}  // namespace lbmk
