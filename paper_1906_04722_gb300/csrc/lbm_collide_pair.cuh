// lbm_collide_pair.cuh -- the collision of collide_core for tau = 1 in both
// components, on component pairs: the two components of every quantity sit in
// one float2 and go through Blackwell's packed FP32 instructions (fma / add /
// mul on two FP32 values per instruction), which halves the arithmetic
// instructions of a kernel that is bound by instruction issue.
//
// At tau = 1 a post-collision population is the equilibrium alone, so of the 19
// pulled pairs only the density and the momentum are needed: a kernel sums them
// (pair_moments) and can drop the populations before it has the neighbours'
// densities.
//
// Bit for bit collide_core<true>: every operation is written with its rounding
// spelled out (which products are fused into the following addition is part of
// the result).  Products with the zero components of e_k are left out, which for
// finite values can change nothing but the sign of a zero.
#pragma once

#include "lbm_device.cuh"

namespace lbmk {

__device__ __forceinline__ float2 pair2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 pmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
// a - b: b times -1 is exact, so the fused form rounds the difference once
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// Densities (Eq. 2, in four interleaved partial sums) and momenta (Eq. 3, over
// opposite pairs) of one cell; at(k) returns the pair (f_k^w, f_k^nw).
template <class At>
__device__ __forceinline__ void pair_moments(At&& at, float2& rho, float2 (&j)[3]) {
    float2 a[4];
    a[0] = at(0);
#pragma unroll
    for (int k = 1; k < Q; k += 2) {
        const float2 p = at(k), m = at(k + 1);
        if (k < 4) a[k] = p;
        else a[k & 3] = padd(a[k & 3], p);
        if (k + 1 < 4) a[k + 1] = m;
        else a[(k + 1) & 3] = padd(a[(k + 1) & 3], m);
        const float2 d = psub(p, m);
        if (k == 1) j[0] = d;
        else if (EX(k)) j[0] = EX(k) > 0 ? padd(j[0], d) : psub(j[0], d);
        if (k == 3) j[1] = d;
        else if (EY(k)) j[1] = EY(k) > 0 ? padd(j[1], d) : psub(j[1], d);
        if (k == 5) j[2] = d;
        else if (EZ(k)) j[2] = EZ(k) > 0 ? padd(j[2], d) : psub(j[2], d);
    }
    rho = padd(padd(a[0], a[1]), padd(a[2], a[3]));
}

// F / r for the three components of F, each quotient correctly rounded:
// Markstein's correction (IBM J. Res. Dev. 34, 1990: with y the correctly
// rounded reciprocal of r and q within one ulp of F / r, q + (F - q r) y rounds
// to the quotient), one reciprocal per component instead of three divisions.
// Densities outside [2^-60, 2^60] take the plain division; 0 for r = 0.
__device__ __forceinline__ void pair_divide(float2 r, const float2 (&F)[3], float2 (&q)[3]) {
    const float lo = 0x1p-60f, hi = 0x1p60f;
    const float ax = fabsf(r.x), ay = fabsf(r.y);
    if (ax >= lo && ax <= hi && ay >= lo && ay <= hi) {
        const float2 y = make_float2(__frcp_rn(r.x), __frcp_rn(r.y));
        const float2 n = make_float2(-r.x, -r.y);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float2 v = pmul(F[d], y);
            v = pfma(pfma(n, v, F[d]), y, v);
            q[d] = pfma(pfma(n, v, F[d]), y, v);
        }
    } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            q[d].x = r.x != 0.f ? __fdiv_rn(F[d].x, r.x) : 0.f;
            q[d].y = r.y != 0.f ? __fdiv_rn(F[d].y, r.y) : 0.f;
        }
    }
}

// Common velocity of both components (densities r, momenta j; the non-wetting
// halves 0 on a membrane cell).
__device__ __forceinline__ void pair_common_velocity(float2 r, const float2 (&j)[3], float (&up)[3]) {
    const float den = __fadd_rn(r.x, r.y);
    const float inv = den != 0.f ? __frcp_rn(den) : 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) up[d] = __fmul_rn(__fadd_rn(j[d].x, j[d].y), inv);
}

// Equilibrium velocities u_eq of both components of a cell with densities r,
// common velocity up and adhesion word a (0: no grain near): cohesion
// (rho_at(k): densities at x + e_k, 0 where that cell is not fluid), adhesion
// and body force.
template <class RhoAt>
__device__ __forceinline__ void pair_velocity(float2 r, const float (&up)[3], uint32_t a, const Phys& P,
                                              RhoAt&& rho_at, float2 (&u)[3]) {
    float2 c[3] = {};
#pragma unroll
    for (int k = 1; k < Q; k += 2) {
        const float2 d = psub(rho_at(k), rho_at(k + 1));
        if (EX(k)) c[0] = pfma(pair2(EX(k) * WK(k)), d, c[0]);
        if (EY(k)) c[1] = pfma(pair2(EY(k) * WK(k)), d, c[1]);
        if (EZ(k)) c[2] = pfma(pair2(EZ(k) * WK(k)), d, c[2]);
    }
    const float2 t1 = pmul(pair2(-P.G), r);
    const float2 t2 = make_float2(__fmul_rn(P.Gads[0], r.x), __fmul_rn(P.Gads[1], r.y));
    float2 F[3], q[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float ad = __fmul_rn((float)(int8_t)((a >> (8 * d)) & 0xffu), 1.0f / 36.0f);
        const float2 b = pmul(t2, pair2(-ad));
        F[d] = pfma(r, pair2(P.g[d]), pfma(t1, make_float2(c[d].y, c[d].x), b));
    }
    pair_divide(r, F, q);
#pragma unroll
    for (int d = 0; d < 3; ++d) u[d] = padd(pair2(up[d]), q[d]);
}

// The 18 moving equilibrium pairs of densities r and velocities u into
// sink(k, pair), and the rest pair rho - (their sum) returned.
template <class Sink>
__device__ __forceinline__ float2 pair_equilibrium(float2 r, const float2 (&u)[3], Sink&& sink) {
    const float2 uu = pfma(u[2], u[2], pfma(u[0], u[0], pmul(u[1], u[1])));
    const float2 base = pmul(r, pfma(pair2(-1.5f), uu, pair2(1.f)));
    const float2 r45 = pmul(pair2(4.5f), r), r3 = pmul(pair2(3.f), r);
    float2 part[3];
#pragma unroll
    for (int k = 1; k < Q; k += 2) {
        float2 e;
        if (k == 1) e = u[0];
        else if (k == 3) e = u[1];
        else if (k == 5) e = u[2];
        else if (EX(k)) e = EY(k) > 0 || EZ(k) > 0 ? padd(u[0], EY(k) ? u[1] : u[2]) : psub(u[0], EY(k) ? u[1] : u[2]);
        else e = EZ(k) > 0 ? padd(u[1], u[2]) : psub(u[1], u[2]);
        const float2 sym = pmul(pair2(WK(k)), pfma(pmul(r45, e), e, base));
        const float2 re = pmul(r3, e);
        const float2 v0 = pfma(pair2(WK(k)), re, sym), v1 = pfma(pair2(-WK(k)), re, sym);
        const float2 s = padd(v0, v1);
        part[(k >> 1) % 3] = k < 6 ? s : padd(part[(k >> 1) % 3], s);
        sink(k, v0);
        sink(k + 1, v1);
    }
    return psub(r, padd(padd(part[0], part[1]), part[2]));
}

// The rest pair of a reservoir cell that holds densities r at rest (its moving
// pairs are pair_equilibrium's at u = 0).  The products are rounded before they
// are added, as collide_core's are; in scalars, because the compiler fuses a
// packed product into a packed addition that follows it.
__device__ __forceinline__ float2 pair_reservoir_rest(float2 r) {
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 1; k < Q; ++k) {
        s.x = __fadd_rn(s.x, __fmul_rn(WK(k), r.x));
        s.y = __fadd_rn(s.y, __fmul_rn(WK(k), r.y));
    }
    return make_float2(__fadd_rn(r.x, -s.x), __fadd_rn(r.y, -s.y));
}

}  // namespace lbmk
