// lbm_step16_pairs.cu -- the two-launch time step of 16-bit storage for tau = 1 in
// both components, on the 16-bit push layout (W[k][cell] holds the pair of
// deviations the cell reads, taken against its density R of the previous step).
//
// The structure of lbm_step_pairs.cu: the first launch rebuilds a cell's
// populations (f = h + w_k R), stores their densities (the new R) and leaves the
// common velocity in three of the cell's own, now dead, words; the second computes
// the equilibria, encodes each against the density of the cell that will hold it,
// feeds the rounding errors into the rest value and pushes the words.  A cell's
// words are rebuilt once, not twice, and the arithmetic runs on component pairs:
// the one-launch push kernel is bound by instruction issue, this one by neither its
// bytes (168 + 32 a cell) nor a march along z (192^3 sample: 433 against 456 us a step,
// 96^3: 46 against 75).  Results equal the staged 16-bit
// kernel's bit for bit.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstring>

#include "lbm_collide_pair.cuh"
#include "lbm_pair16.cuh"

namespace lbmk {

namespace {

constexpr int PAIR16_THREADS = 128;

template <class H2>
__global__ void __launch_bounds__(PAIR16_THREADS, 8)
    pair16_moment_kernel(uint32_t* __restrict__ W, const float2* __restrict__ Rin, float2* __restrict__ rho,
                         const uint32_t* __restrict__ nbr, int plane, int N) {
    const int c = blockIdx.x * PAIR16_THREADS + threadIdx.x;
    if (c >= N) return;
    const uint32_t cls = (__ldg(nbr + c) >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    const bool has_nw = cls != CLS_MEMBRANE;  // there the non-wetting half of a word may hold anything
    uint32_t u[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) u[k] = __ldcs(W + (size_t)k * plane + c);
    const float2 R = __ldcs(Rin + c);
    float2 r, j[3];
    float up[3];
    pair_moments(
        [&](int k) {
            const float2 f = pfma(pair2(WK(k)), R, Pair<H2>::unpack(u[k]));
            return has_nw ? f : make_float2(f.x, 0.f);
        },
        r, j);
    pair_common_velocity(r, j, up);
    rho[c] = r;
#pragma unroll
    for (int d = 0; d < 3; ++d) W[(size_t)d * plane + c] = __float_as_uint(up[d]);
}

// LARGE: from PAIR16_LARGE cells on the launch waits for its scattered stores, and more
// warps with the neighbour densities read twice (from L1) are the faster form; on
// smaller boxes, which wait for the first loads, they stay in registers (4 CTAs of
// 128 threads an SM instead of 7).  Registers against twice read, us a step: 32^3 4.7 /
// 5.5, 64^3 14.2 / 15.3, 96^3 41.1 / 42.8, 104^3 53.9 / 54.6, 112^3 70.6 / 70.2, 128^3
// 115 / 110, 160^3 238 / 224 (a third of grains: 84^3 30.8 / 31.3, 92^3 42.0 / 41.0,
// 112^3 79.8 / 76.6).
constexpr int PAIR16_LARGE = 1 << 20;

template <class H2, bool LARGE>
__global__ void __launch_bounds__(PAIR16_THREADS, LARGE ? 7 : 4)
    pair16_push_kernel(const uint32_t* __restrict__ W, uint32_t* __restrict__ out, const float2* __restrict__ rho,
                       const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw,
                       const uint32_t* __restrict__ adh, Geom g, Phys P, int N) {
    const int c = blockIdx.x * PAIR16_THREADS + threadIdx.x;
    if (c >= N) return;
    const int row = c / g.nx, x = c - row * g.nx, z = row / g.ny, y = row - z * g.ny;
    // steps to the neighbours in cells, wrapped on every axis (beyond a closed edge the
    // wall bit is set and the step not taken); every load goes out at once
    const int xp = x == g.nx - 1 ? 1 - g.nx : 1, xm = x == 0 ? g.nx - 1 : -1;
    const int yp = y == g.ny - 1 ? g.nx - g.nxy : g.nx, ym = y == 0 ? g.nxy - g.nx : -g.nx;
    const int zp = z == g.nz - 1 ? g.nxy - N : g.nxy, zm = z == 0 ? N - g.nxy : -g.nxy;
    auto step = [&](int k) {
        return (EX(k) > 0 ? xp : EX(k) < 0 ? xm : 0) + (EY(k) > 0 ? yp : EY(k) < 0 ? ym : 0) +
               (EZ(k) > 0 ? zp : EZ(k) < 0 ? zm : 0);
    };
    const uint32_t w = __ldg(nbr + c);
    const float2 self = __ldg(rho + c);
    float up[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) up[d] = __uint_as_float(__ldcs(W + (size_t)d * g.plane + c));
    float2 held[Q];
    if constexpr (!LARGE) {
#pragma unroll
        for (int k = 1; k < Q; ++k) held[k] = __ldg(rho + c + step(k));
    }
    auto nb = [&](int k) { return LARGE ? __ldg(rho + c + step(k)) : held[k]; };
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    float2 r = self, u[3], rest;
    const bool open_end = cls == CLS_INLET || cls == CLS_OUTLET;
    if (open_end) {
        const float* b = P.bc + (cls == CLS_INLET ? 0 : 2);
        r = make_float2(__ldg(b), __ldg(b + 1));
        u[0] = u[1] = u[2] = make_float2(0.f, 0.f);
        rest = pair_reservoir_rest(r);
    } else {
        const uint32_t ad = (w & BIT_ADH) ? __ldg(adh + c) : 0u;
        pair_velocity(r, up, ad, P,
                      [&](int k) { return (w >> OPP(k)) & 1u ? make_float2(0.f, 0.f) : nb(k); }, u);
    }
    // word of the cell that direction k streams to, or the own opposite word at a wall
    auto target = [&](int k, uint32_t bits) {
        return ((bits >> OPP(k)) & 1u) ? (size_t)OPP(k) * g.plane + c : (size_t)k * g.plane + c + step(k);
    };
    float2 err = make_float2(0.f, 0.f), sum;
    const bool has_nw = cls != CLS_MEMBRANE;
    if (has_nw && !(w & BIT_NW_DIFF)) {
        sum = pair_equilibrium(r, u, [&](int k, float2 v) {
            const float2 d = (w >> OPP(k)) & 1u ? self : nb(k);
            const float2 e = pfma(pair2(-WK(k)), d, v);
            const uint32_t h = Pair<H2>::pack(e.x, e.y);
            err = padd(err, psub(e, Pair<H2>::unpack(h)));
            out[target(k, w)] = h;
        });
    } else {  // the components part ways near a membrane
        const uint32_t wn = has_nw ? __ldg(nbr_nw + c) : 0u;
        unsigned short* o16 = reinterpret_cast<unsigned short*>(out);
        sum = pair_equilibrium(r, u, [&](int k, float2 v) {
            const float dw = (w >> OPP(k)) & 1u ? self.x : nb(k).x;
            const float dn = (wn >> OPP(k)) & 1u ? self.y : nb(k).y;
            const float2 e = make_float2(__fmaf_rn(-WK(k), dw, v.x), has_nw ? __fmaf_rn(-WK(k), dn, v.y) : 0.f);
            const uint32_t h = Pair<H2>::pack(e.x, e.y);
            err = padd(err, psub(e, Pair<H2>::unpack(h)));
            o16[2 * target(k, w)] = (unsigned short)(h & 0xffffu);
            if (has_nw) o16[2 * target(k, wn) + 1] = (unsigned short)(h >> 16);
        });
    }
    if (open_end) sum = rest;
    const float2 e0 = padd(pfma(pair2(-WK(0)), self, sum), err);
    out[c] = Pair<H2>::pack(e0.x, has_nw ? e0.y : 0.f);
}

}  // namespace

template <class H2>
static cudaError_t launch_pairs16(uint32_t* win, uint32_t* wout, const float2* Rin, float2* Rout, const uint32_t* nbr,
                                  const uint32_t* nbr_nw, const uint32_t* adh, const Geom& g, const Phys& p,
                                  cudaStream_t s) {
    const int N = g.nxy * g.nz;
    const unsigned blocks = (unsigned)((N + PAIR16_THREADS - 1) / PAIR16_THREADS);
    pair16_moment_kernel<H2><<<blocks, PAIR16_THREADS, 0, s>>>(win, Rin, Rout, nbr, g.plane, N);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (N >= PAIR16_LARGE)
        pair16_push_kernel<H2, true><<<blocks, PAIR16_THREADS, 0, s>>>(win, wout, Rout, nbr, nbr_nw, adh, g, p, N);
    else
        pair16_push_kernel<H2, false><<<blocks, PAIR16_THREADS, 0, s>>>(win, wout, Rout, nbr, nbr_nw, adh, g, p, N);
    return cudaGetLastError();
}

cudaError_t launch_step16_pairs(int precision, uint32_t* win, uint32_t* wout, const float2* Rin, float2* Rout,
                                const uint32_t* nbr, const uint32_t* nbr_nw, const uint32_t* adh, const Geom& g,
                                const Phys& p, cudaStream_t s) {
    return precision == 1 ? launch_pairs16<__half2>(win, wout, Rin, Rout, nbr, nbr_nw, adh, g, p, s)
                          : launch_pairs16<__nv_bfloat162>(win, wout, Rin, Rout, nbr, nbr_nw, adh, g, p, s);
}

}  // namespace lbmk
