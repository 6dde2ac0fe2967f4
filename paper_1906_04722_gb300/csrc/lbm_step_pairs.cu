// lbm_step_pairs.cu -- the two-launch time step on the paired push layout (float2
// F[nz][ny][19][nx], a cell's populations at the current time level at its own
// address), in a form for tau = 1 in both components and a general one.
//
// At tau = 1 the collision needs a cell's density and momentum only.  The first
// launch reads a cell's 19 pairs once and leaves its densities (8 bytes, compact)
// and common velocity (12 bytes, in two of the cell's own, now dead, slots); the
// second computes the equilibria from those and the neighbours' densities and
// pushes them.  There is no shared memory, no barrier and no serial march along z,
// so a small box is two short latencies instead of a chain of planes: a step of a
// 32^3 throat takes 4.2 us (staged kernel 10.4), of a 48^3 periodic box 7.1 us
// (16.1).  On the 192^3 sample the first launch streams at 6.5 TB/s (178 us, its
// 1.16 GB are whole rows with their grain) and the second, which waits on its
// scattered 8-byte stores (47 M partial sectors for 25 M), takes 0.30 ms at 3.8
// TB/s: 0.49 ms a step against 0.42 of the tuned push kernel and 0.69 of the staged
// one; boxes of that size step on moments (lbm_step_moments.cu). 
//
// At any other tau the populations count as well: the first launch leaves the
// densities only and the second reads the 19 pairs again (out of L2 while the two
// buffers fit there), collides with collide_core and pushes.  Periodic open boxes at
// tau = 0.8 and 1.2, a step (staged kernel; the two launches on the pull layout that
// this form replaced): 16^3 4.3 us (8.7; 7.4), 32^3 5.0 (10.5; 7.8), 48^3 9.5 (16.2;
// 15.2), 64^3 15.7 (35.0; 25.5), 101 x 90 x 77 48 (78; 100), 128^3 147 (245; 230),
// 192^3 507 (647; 759).  A third of grains changes little (192^3: 511 against 659).
//
// Any box and any periodic axes; results equal the staged kernel's bit for bit.
#include "lbm_collide_pair.cuh"
#include "lbm_step_core.cuh"

namespace lbmk {

namespace {

constexpr int PAIR_THREADS = 128;

// Slot 0 of cell c (c = row nx + x) in the paired layout; slot k lies k nx further.
__device__ __forceinline__ int slot0(int c, int row, const Geom& g) { return c + row * (Q - 1) * g.nx; }

// The steps to a cell's neighbours in cells, wrapped on every axis: inside the box
// whatever the axis is (beyond a closed edge the wall bit is set and the step not taken).
struct Around {
    int s0, nx, xp, xm, yp, ym, zp, zm;
    __device__ __forceinline__ Around(int c, const Geom& g, int N) {
        const int row = c / g.nx, x = c - row * g.nx, z = row / g.ny, y = row - z * g.ny;
        s0 = slot0(c, row, g);
        nx = g.nx;
        xp = x == g.nx - 1 ? 1 - g.nx : 1, xm = x == 0 ? g.nx - 1 : -1;
        yp = y == g.ny - 1 ? g.nx - g.nxy : g.nx, ym = y == 0 ? g.nxy - g.nx : -g.nx;
        zp = z == g.nz - 1 ? g.nxy - N : g.nxy, zm = z == 0 ? N - g.nxy : -g.nxy;
    }
    __device__ __forceinline__ int dx(int k) const { return EX(k) > 0 ? xp : EX(k) < 0 ? xm : 0; }
    __device__ __forceinline__ int dr(int k) const {
        return (EY(k) > 0 ? yp : EY(k) < 0 ? ym : 0) + (EZ(k) > 0 ? zp : EZ(k) < 0 ? zm : 0);
    }
    // slot of the cell that direction k streams to, or the own opposite slot at a wall
    __device__ __forceinline__ int target(int k, uint32_t bits) const {
        return ((bits >> OPP(k)) & 1u) ? s0 + OPP(k) * nx : s0 + k * nx + dx(k) + Q * dr(k);
    }
};

// MOMENTS: leave the common velocity at tau = 1 too, in the populations' place.
template <bool MOMENTS>
__global__ void __launch_bounds__(PAIR_THREADS, 8)
    pair_moment_kernel(float2* __restrict__ F, float2* __restrict__ rho2, const uint32_t* __restrict__ nbr, Geom g,
                       int N) {
    const int c = blockIdx.x * PAIR_THREADS + threadIdx.x;
    if (c >= N) return;
    const uint32_t cls = (__ldg(nbr + c) >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    float2* f = F + slot0(c, c / g.nx, g);
    float2 v[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) v[k] = __ldcs(f + k * g.nx);
    const bool has_nw = cls != CLS_MEMBRANE;  // there the non-wetting half of a slot may hold anything
    float2 r, j[3];
    float up[3];
    pair_moments([&](int k) { return has_nw ? v[k] : make_float2(v[k].x, 0.f); }, r, j);
    rho2[c] = r;
    if constexpr (MOMENTS) {
        pair_common_velocity(r, j, up);
        f[0] = make_float2(up[0], up[1]);
        f[g.nx] = make_float2(up[2], 0.f);
    }
}

__global__ void __launch_bounds__(PAIR_THREADS, 8)
    pair_push_kernel(const float2* __restrict__ F, float2* __restrict__ out, const float2* __restrict__ rho2,
                     const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw,
                     const uint32_t* __restrict__ adh, Geom g, Phys P, int N) {
    const int c = blockIdx.x * PAIR_THREADS + threadIdx.x;
    if (c >= N) return;
    const Around at(c, g, N);
    const int s0 = at.s0;
    // The launch waits for memory, so every load goes out at once, before the
    // geometry word says which of them count (a wall's density, which may be
    // anything, is replaced by 0): 4.6 -> 4.2 us a step of a 32^3 throat.
    const uint32_t w = __ldg(nbr + c);
    float2 r = __ldg(rho2 + c), u[3], rest;
    const float2 va = __ldcs(F + s0), vb = __ldcs(F + s0 + g.nx);
    float2 nb[Q];
#pragma unroll
    for (int k = 1; k < Q; ++k) nb[k] = __ldg(rho2 + c + at.dx(k) + at.dr(k));
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    const bool open_end = cls == CLS_INLET || cls == CLS_OUTLET;
    if (open_end) {
        const float* b = P.bc + (cls == CLS_INLET ? 0 : 2);
        r = make_float2(__ldg(b), __ldg(b + 1));
        u[0] = u[1] = u[2] = make_float2(0.f, 0.f);
        rest = pair_reservoir_rest(r);
    } else {
        const float up[3] = {va.x, va.y, vb.x};
        const uint32_t ad = (w & BIT_ADH) ? __ldg(adh + c) : 0u;
        pair_velocity(r, up, ad, P,
                      [&](int k) { return (w >> OPP(k)) & 1u ? make_float2(0.f, 0.f) : nb[k]; }, u);
    }
    float2 sum;
    if (cls == CLS_MEMBRANE || (w & BIT_NW_DIFF)) {  // the components part ways near a membrane
        const bool has_nw = cls != CLS_MEMBRANE;
        const uint32_t wn = has_nw ? __ldg(nbr_nw + c) : 0u;
        sum = pair_equilibrium(r, u, [&](int k, float2 v) {
            out[at.target(k, w)].x = v.x;
            if (has_nw) out[at.target(k, wn)].y = v.y;
        });
        out[s0].x = open_end ? rest.x : sum.x;
        if (has_nw) out[s0].y = open_end ? rest.y : sum.y;
    } else {
        sum = pair_equilibrium(r, u, [&](int k, float2 v) { out[at.target(k, w)] = v; });
        out[s0] = open_end ? rest : sum;
    }
}

// The second launch for any tau.  Like the first it waits for memory: all loads go
// out before the geometry word says which of them count.
__global__ void __launch_bounds__(PAIR_THREADS, 5)
    pair_relax_kernel(const float2* __restrict__ F, float2* __restrict__ out, const float2* __restrict__ rho2,
                      const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw,
                      const uint32_t* __restrict__ adh, Geom g, Phys P, int N) {
    const int c = blockIdx.x * PAIR_THREADS + threadIdx.x;
    if (c >= N) return;
    const Around at(c, g, N);
    const uint32_t w = __ldg(nbr + c);
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    float2 nb[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) nb[k] = __ldg(rho2 + c + at.dx(k) + at.dr(k));
    const bool has_nw = cls != CLS_MEMBRANE;
    float f[2][Q], o[2][Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const float2 v = __ldcs(F + at.s0 + k * g.nx);
        f[0][k] = v.x;
        f[1][k] = has_nw ? v.y : 0.f;
    }
    const uint32_t ad = (w & BIT_ADH) ? __ldg(adh + c) : 0u;
    collide_core(
        f, w, ad, P, [&](int k) { return k && ((w >> OPP(k)) & 1u) ? make_float2(0.f, 0.f) : nb[k]; },
        [&](int s, int k, float v) { o[s][k] = v; });
    if (!has_nw || (w & BIT_NW_DIFF)) {  // the components part ways near a membrane
        const uint32_t wn = has_nw ? __ldg(nbr_nw + c) : 0u;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            out[k ? at.target(k, w) : at.s0].x = o[0][k];
            if (has_nw) out[k ? at.target(k, wn) : at.s0].y = o[1][k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < Q; ++k) out[k ? at.target(k, w) : at.s0] = make_float2(o[0][k], o[1][k]);
    }
}

}  // namespace

bool pair_step_applicable(const Phys& p) { return p.tau[0] == 1.0f && p.tau[1] == 1.0f; }

cudaError_t launch_pair_moments(float* F, float2* rho2, const uint32_t* nbr, const Geom& g, cudaStream_t s) {
    const int N = g.nxy * g.nz;
    pair_moment_kernel<true><<<(unsigned)((N + PAIR_THREADS - 1) / PAIR_THREADS), PAIR_THREADS, 0, s>>>(
        reinterpret_cast<float2*>(F), rho2, nbr, g, N);
    return cudaGetLastError();
}

cudaError_t launch_step_pairs(float* fin, float* fout, float2* rho2, const uint32_t* nbr, const uint32_t* nbr_nw,
                              const uint32_t* adh, const Geom& g, const Phys& p, cudaStream_t s) {
    const int N = g.nxy * g.nz;
    const unsigned blocks = (unsigned)((N + PAIR_THREADS - 1) / PAIR_THREADS);
    if (!pair_step_applicable(p)) {
        pair_moment_kernel<false><<<blocks, PAIR_THREADS, 0, s>>>(reinterpret_cast<float2*>(fin), rho2, nbr, g, N);
        pair_relax_kernel<<<blocks, PAIR_THREADS, 0, s>>>(reinterpret_cast<const float2*>(fin),
                                                          reinterpret_cast<float2*>(fout), rho2, nbr, nbr_nw, adh, g,
                                                          p, N);
        return cudaGetLastError();
    }
    cudaError_t e = launch_pair_moments(fin, rho2, nbr, g, s);
    if (e != cudaSuccess) return e;
    pair_push_kernel<<<blocks, PAIR_THREADS, 0, s>>>(reinterpret_cast<const float2*>(fin),
                                                    reinterpret_cast<float2*>(fout), rho2, nbr, nbr_nw, adh, g, p, N);
    return cudaGetLastError();
}

}  // namespace lbmk
