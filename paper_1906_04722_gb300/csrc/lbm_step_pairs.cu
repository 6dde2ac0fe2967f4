// lbm_step_pairs.cu -- the two-launch time step for tau = 1 in both components, on
// the paired push layout (float2 F[nz][ny][19][nx], a cell's populations at the
// current time level at its own address).
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
// one; boxes of that size step on moments (lbm_step_moments.cu).  Any box and any periodic axes; results equal the staged kernel's bit for bit.
#include "lbm_collide_pair.cuh"

namespace lbmk {

namespace {

constexpr int PAIR_THREADS = 128;

// Slot 0 of cell c (c = row nx + x) in the paired layout; slot k lies k nx further.
__device__ __forceinline__ int slot0(int c, int row, const Geom& g) { return c + row * (Q - 1) * g.nx; }

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
    pair_common_velocity(r, j, up);
    rho2[c] = r;
    f[0] = make_float2(up[0], up[1]);
    f[g.nx] = make_float2(up[2], 0.f);
}

__global__ void __launch_bounds__(PAIR_THREADS, 8)
    pair_push_kernel(const float2* __restrict__ F, float2* __restrict__ out, const float2* __restrict__ rho2,
                     const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw,
                     const uint32_t* __restrict__ adh, Geom g, Phys P, int N) {
    const int c = blockIdx.x * PAIR_THREADS + threadIdx.x;
    if (c >= N) return;
    const int row = c / g.nx, x = c - row * g.nx, z = row / g.ny, y = row - z * g.ny;
    const int s0 = slot0(c, row, g);
    // steps to the neighbours in cells, wrapped on every axis: inside the box whatever
    // the axis is (beyond a closed edge the wall bit is set and the step not taken)
    const int xp = x == g.nx - 1 ? 1 - g.nx : 1, xm = x == 0 ? g.nx - 1 : -1;
    const int yp = y == g.ny - 1 ? g.nx - g.nxy : g.nx, ym = y == 0 ? g.nxy - g.nx : -g.nx;
    const int zp = z == g.nz - 1 ? g.nxy - N : g.nxy, zm = z == 0 ? N - g.nxy : -g.nxy;
    auto dx = [&](int k) { return EX(k) > 0 ? xp : EX(k) < 0 ? xm : 0; };
    auto dr = [&](int k) {
        return (EY(k) > 0 ? yp : EY(k) < 0 ? ym : 0) + (EZ(k) > 0 ? zp : EZ(k) < 0 ? zm : 0);
    };
    // The launch waits for memory, so every load goes out at once, before the
    // geometry word says which of them count (a wall's density, which may be
    // anything, is replaced by 0): 4.6 -> 4.2 us a step of a 32^3 throat.
    const uint32_t w = __ldg(nbr + c);
    float2 r = __ldg(rho2 + c), u[3], rest;
    const float2 va = __ldcs(F + s0), vb = __ldcs(F + s0 + g.nx);
    float2 nb[Q];
#pragma unroll
    for (int k = 1; k < Q; ++k) nb[k] = __ldg(rho2 + c + dx(k) + dr(k));
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
    // slot of the cell that direction k streams to, or the own opposite slot at a wall
    auto target = [&](int k, uint32_t bits) {
        return ((bits >> OPP(k)) & 1u) ? s0 + OPP(k) * g.nx : s0 + k * g.nx + dx(k) + Q * dr(k);
    };
    float2 sum;
    if (cls == CLS_MEMBRANE || (w & BIT_NW_DIFF)) {  // the components part ways near a membrane
        const bool has_nw = cls != CLS_MEMBRANE;
        const uint32_t wn = has_nw ? __ldg(nbr_nw + c) : 0u;
        sum = pair_equilibrium(r, u, [&](int k, float2 v) {
            out[target(k, w)].x = v.x;
            if (has_nw) out[target(k, wn)].y = v.y;
        });
        out[s0].x = open_end ? rest.x : sum.x;
        if (has_nw) out[s0].y = open_end ? rest.y : sum.y;
    } else {
        sum = pair_equilibrium(r, u, [&](int k, float2 v) { out[target(k, w)] = v; });
        out[s0] = open_end ? rest : sum;
    }
}

}  // namespace

bool pair_step_applicable(const Phys& p) { return p.tau[0] == 1.0f && p.tau[1] == 1.0f; }

cudaError_t launch_pair_moments(float* F, float2* rho2, const uint32_t* nbr, const Geom& g, cudaStream_t s) {
    const int N = g.nxy * g.nz;
    pair_moment_kernel<<<(unsigned)((N + PAIR_THREADS - 1) / PAIR_THREADS), PAIR_THREADS, 0, s>>>(
        reinterpret_cast<float2*>(F), rho2, nbr, g, N);
    return cudaGetLastError();
}

cudaError_t launch_step_pairs(float* fin, float* fout, float2* rho2, const uint32_t* nbr, const uint32_t* nbr_nw,
                              const uint32_t* adh, const Geom& g, const Phys& p, cudaStream_t s) {
    const int N = g.nxy * g.nz;
    const unsigned blocks = (unsigned)((N + PAIR_THREADS - 1) / PAIR_THREADS);
    cudaError_t e = launch_pair_moments(fin, rho2, nbr, g, s);
    if (e != cudaSuccess) return e;
    pair_push_kernel<<<blocks, PAIR_THREADS, 0, s>>>(reinterpret_cast<const float2*>(fin),
                                                    reinterpret_cast<float2*>(fout), rho2, nbr, nbr_nw, adh, g, p, N);
    return cudaGetLastError();
}

}  // namespace lbmk
