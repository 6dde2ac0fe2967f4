// lbm_step_moments.cu -- the FP32 time step for tau = 1 in both components on
// moments: 48 bytes a cell instead of 152.
//
// At tau = 1 a post-collision population is an equilibrium, a function of ten
// numbers a cell (both components' density, velocity and rest population).  So the
// state need not be kept as populations at all: a cell's incoming populations are
// computed from its neighbours' moments, with the very operations that would have
// stored them (pair_equilibrium's, one direction at a time), and agree bit for bit.
//
//   moment_gather_kernel   reads the neighbours' moments (rs, base, u, rest), forms
//                          the 19 incoming pairs, and stores the cell's densities
//                          and common velocity (20 bytes);
//   moment_collide_kernel  reads those and the neighbours' densities and stores the
//                          cell's new moments (48 bytes).
//
// Each launch reads what the other wrote, so one copy of the state is enough; it
// lies in one population buffer.  DRAM moves about 0.9 GB a step of the 192^3 sample,
// where the tuned push kernel moves 2.1; the price is arithmetic (each direction's
// equilibrium is formed by its reader, without the sharing between opposite
// directions) and loads, which L1 and L2 serve.  Bound by the latency of those
// loads: a CTA is a 32 x 4 x 2 brick, six to an SM (40 registers a thread), and a
// cell's densities and u^2 term come in one 16-byte load.  192^3: 319 us a step (420
// push kernel, 492 on pairs); bricks of 32 x 2 x 2 at eight an SM (64 registers) 370,
// 32 x 4 x 1 at twelve 321, 32 x 8 x 2 at two 389.
#include "lbm_collide_pair.cuh"

namespace lbmk {

namespace {

constexpr int MX = MOMENT_ROW, MY = 4, MZ = 2, MT = MX * MY * MZ;

// Arrays of the state in a population buffer, `plane` pairs apart.
struct Moments {
    float4* rb;          // equilibrium densities rs and rs (1 - 1.5 u^2), the components side by side
    float2 *u[3], *rest;  // equilibrium velocity, rest pair
    float2 *rho, *upxy;   // densities of the cells and their common velocity
    float* upz;
};
__host__ __device__ __forceinline__ Moments moments_in(float* buffer, int plane) {
    float2* b = reinterpret_cast<float2*>(buffer);
    Moments m;
    m.rb = reinterpret_cast<float4*>(buffer);
    for (int d = 0; d < 3; ++d) m.u[d] = b + (size_t)(2 + d) * plane;
    m.rest = b + (size_t)5 * plane;
    m.rho = b + (size_t)6 * plane;
    m.upxy = b + (size_t)7 * plane;
    m.upz = reinterpret_cast<float*>(b + (size_t)8 * plane);
    return m;
}

// Cell (x, y, z) with its steps to the neighbours, wrapped on every axis (beyond a
// closed edge the wall bit is set and the step not taken).
struct Cell {
    int c, xp, xm, yp, ym, zp, zm;
    __device__ __forceinline__ Cell(int x, int y, int z, const Geom& g) {
        const int N = g.nxy * g.nz;
        c = z * g.nxy + y * g.nx + x;
        xp = x == g.nx - 1 ? 1 - g.nx : 1;
        xm = x == 0 ? g.nx - 1 : -1;
        yp = y == g.ny - 1 ? g.nx - g.nxy : g.nx;
        ym = y == 0 ? g.nxy - g.nx : -g.nx;
        zp = z == g.nz - 1 ? g.nxy - N : g.nxy;
        zm = z == 0 ? N - g.nxy : -g.nxy;
    }
    __device__ __forceinline__ int to(int k) const {  // the cell at x + e_k
        return c + (EX(k) > 0 ? xp : EX(k) < 0 ? xm : 0) + (EY(k) > 0 ? yp : EY(k) < 0 ? ym : 0) +
               (EZ(k) > 0 ? zp : EZ(k) < 0 ? zm : 0);
    }
};

// What cell s sends in direction k (reversed: in direction opposite to k).
__device__ __forceinline__ float2 sent(const Moments& m, int s, int k, bool reversed) {
    const int o = k & 1 ? k : k - 1;  // the odd direction of the pair
    const float4 rb = __ldg(m.rb + s);
    const float2 r = make_float2(rb.x, rb.y), base = make_float2(rb.z, rb.w);
    const float2 ux = EX(o) ? __ldg(m.u[0] + s) : make_float2(0.f, 0.f);
    const float2 uy = EY(o) ? __ldg(m.u[1] + s) : make_float2(0.f, 0.f);
    const float2 uz = EZ(o) ? __ldg(m.u[2] + s) : make_float2(0.f, 0.f);
    float2 e;
    if (o == 1) e = ux;
    else if (o == 3) e = uy;
    else if (o == 5) e = uz;
    else if (EX(o)) e = EY(o) > 0 || EZ(o) > 0 ? padd(ux, EY(o) ? uy : uz) : psub(ux, EY(o) ? uy : uz);
    else e = EZ(o) > 0 ? padd(uy, uz) : psub(uy, uz);
    const float2 sym = pmul(pair2(WK(k)), pfma(pmul(pmul(pair2(4.5f), r), e), e, base));
    const float2 re = pmul(pmul(pair2(3.f), r), e);
    const float sign = ((k & 1) != 0) != reversed ? WK(k) : -WK(k);
    return pfma(pair2(sign), re, sym);
}

// The pair that arrives at the cell in direction k: sent by x - e_k, or reflected
// where that is not fluid for the component (w, wn: bounce bits of the two).
__device__ __forceinline__ float2 arriving(const Moments& m, const Cell& at, int k, uint32_t w, uint32_t wn,
                                           bool split) {
    if (k == 0) return __ldg(m.rest + at.c);
    const bool wall = (w >> k) & 1u;
    float2 v = sent(m, wall ? at.c : at.to(OPP(k)), k, wall);
    if (split) {  // next to a membrane the components' walls differ
        const bool wall_n = (wn >> k) & 1u;
        if (wall_n != wall) v.y = sent(m, wall_n ? at.c : at.to(OPP(k)), k, wall_n).y;
    }
    return v;
}

__device__ __forceinline__ bool my_cell(const Geom& g, int& x, int& y, int& z) {
    x = blockIdx.x * MX + threadIdx.x;
    y = blockIdx.y * MY + threadIdx.y;
    z = blockIdx.z * MZ + threadIdx.z;
    return x < g.nx && y < g.ny && z < g.nz;
}

__global__ void __launch_bounds__(MT, 6)
    moment_gather_kernel(float* buffer, const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw, Geom g) {
    int x, y, z;
    if (!my_cell(g, x, y, z)) return;
    const Cell at(x, y, z, g);
    const uint32_t w = __ldg(nbr + at.c);
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    const Moments m = moments_in(buffer, g.plane);
    const bool has_nw = cls != CLS_MEMBRANE, split = has_nw && (w & BIT_NW_DIFF);
    const uint32_t wn = split ? __ldg(nbr_nw + at.c) : w;
    float2 r, j[3];
    float up[3];
    pair_moments(
        [&](int k) {
            const float2 v = arriving(m, at, k, w, wn, split);
            return has_nw ? v : make_float2(v.x, 0.f);
        },
        r, j);
    pair_common_velocity(r, j, up);
    m.rho[at.c] = r;
    m.upxy[at.c] = make_float2(up[0], up[1]);
    m.upz[at.c] = up[2];
}

// FIRST: the densities and common velocity come from a step that started on
// populations (pair_moment_kernel: rho2, and two of the cell's slots in F).
template <bool FIRST>
__global__ void __launch_bounds__(MT, 6)
    moment_collide_kernel(float* buffer, const float2* __restrict__ F, const float2* __restrict__ rho2,
                          const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ adh, Geom g, Phys P) {
    int x, y, z;
    if (!my_cell(g, x, y, z)) return;
    const Cell at(x, y, z, g);
    const Moments m = moments_in(buffer, g.plane);
    const float2* rho = FIRST ? rho2 : m.rho;
    const uint32_t w = __ldg(nbr + at.c), ad = __ldg(adh + at.c);
    const int slot = at.c + (z * g.ny + y) * (Q - 1) * g.nx;
    const float2 a = FIRST ? __ldg(F + slot) : __ldg(m.upxy + at.c);
    const float up[3] = {a.x, a.y, FIRST ? __ldg(F + slot + g.nx).x : __ldg(m.upz + at.c)};
    float2 r = __ldg(rho + at.c), u[3], rest;
    const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
    if (cls == CLS_SOLID) return;
    const bool open_end = cls == CLS_INLET || cls == CLS_OUTLET;
    if (open_end) {
        const float* b = P.bc + (cls == CLS_INLET ? 0 : 2);
        r = make_float2(__ldg(b), __ldg(b + 1));
        u[0] = u[1] = u[2] = make_float2(0.f, 0.f);
        rest = pair_reservoir_rest(r);
    } else {
        pair_velocity(r, up, (w & BIT_ADH) ? ad : 0u, P,
                      [&](int k) {
                          const bool wall = (w >> OPP(k)) & 1u;
                          const float2 v = __ldg(rho + (wall ? at.c : at.to(k)));
                          return wall ? make_float2(0.f, 0.f) : v;
                      },
                      u);
    }
    const float2 sum = pair_equilibrium(r, u, [](int, float2) {});
    if (!open_end) rest = sum;
    // pair_equilibrium's own u^2 and base
    const float2 uu = pfma(u[2], u[2], pfma(u[0], u[0], pmul(u[1], u[1])));
    const float2 base = pmul(r, pfma(pair2(-1.5f), uu, pair2(1.f)));
    m.rb[at.c] = make_float4(r.x, r.y, base.x, base.y);
#pragma unroll
    for (int d = 0; d < 3; ++d) m.u[d][at.c] = u[d];
    m.rest[at.c] = rest;
}

// Densities of a cell, summed in k order as the read-outs of the other layouts.
__device__ __forceinline__ float2 moment_density(const Moments& m, const Cell& at, uint32_t w,
                                                 const uint32_t* __restrict__ nbr_nw) {
    const bool has_nw = ((w >> CLS_SHIFT) & CLS_MASK) != CLS_MEMBRANE, split = has_nw && (w & BIT_NW_DIFF);
    const uint32_t wn = split ? __ldg(nbr_nw + at.c) : w;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < Q; ++k) s = padd(s, arriving(m, at, k, w, wn, split));
    return has_nw ? s : make_float2(s.x, 0.f);
}

// The density field as pairs (0 where a component is not fluid).
__global__ void __launch_bounds__(MT)
    moment_density_kernel(float* buffer, const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ nbr_nw, Geom g,
                          float2* __restrict__ rho2) {
    int x, y, z;
    if (!my_cell(g, x, y, z)) return;
    const Cell at(x, y, z, g);
    const uint32_t w = __ldg(nbr + at.c);
    const bool solid = ((w >> CLS_SHIFT) & CLS_MASK) == CLS_SOLID;
    rho2[at.c] = solid ? make_float2(0.f, 0.f) : moment_density(moments_in(buffer, g.plane), at, w, nbr_nw);
}

__global__ void moment_probe_kernel(float* buffer, const uint32_t* __restrict__ nbr,
                                    const uint32_t* __restrict__ nbr_nw, Geom g, int x, int y, int z, float* out) {
    const Cell at(x, y, z, g);
    const uint32_t w = __ldg(nbr + at.c);
    const bool solid = ((w >> CLS_SHIFT) & CLS_MASK) == CLS_SOLID;
    const float2 r = solid ? make_float2(0.f, 0.f) : moment_density(moments_in(buffer, g.plane), at, w, nbr_nw);
    out[0] = r.x;
    out[1] = r.y;
}

// Read-outs of a density field of pairs.
__global__ void split_density_kernel(const float2* __restrict__ rho2, float* __restrict__ rho, long long N) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float2 r = rho2[c];
        rho[c] = r.x;
        rho[N + c] = r.y;
    }
}
__global__ void __launch_bounds__(256)
    measure_density_kernel(const float2* __restrict__ rho2, const uint32_t* __restrict__ nbr, long long N, double G,
                           double* __restrict__ partials) {
    MeasureSums sums;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const float2 r = __ldg(rho2 + c);
        sums.add((__ldg(nbr + c) >> CLS_SHIFT) & CLS_MASK, r.x, r.y, G);
    }
    sums.store<8>(partials + (size_t)blockIdx.x * NMEAS);
}

// Moments -> pull layout: the post-collision populations of every cell at the cell.
__global__ void __launch_bounds__(MT)
    moments_to_pull_kernel(float* buffer, float* __restrict__ fout, const uint32_t* __restrict__ nbr, Geom g) {
    int x, y, z;
    if (!my_cell(g, x, y, z)) return;
    const int c = z * g.nxy + y * g.nx + x;
    const uint32_t cls = (__ldg(nbr + c) >> CLS_SHIFT) & CLS_MASK;
    const Moments m = moments_in(buffer, g.plane);
    const bool fluid = cls != CLS_SOLID, has_nw = fluid && cls != CLS_MEMBRANE;
    const float2 zero = make_float2(0.f, 0.f);
    const float2 r = fluid ? make_float2(m.rb[c].x, m.rb[c].y) : zero, rest = fluid ? m.rest[c] : zero;
    const float2 u[3] = {fluid ? m.u[0][c] : zero, fluid ? m.u[1][c] : zero, fluid ? m.u[2][c] : zero};
    auto put = [&](int k, float2 v) {
        fout[(size_t)k * g.plane + c] = fluid ? v.x : 0.f;
        fout[(size_t)(Q + k) * g.plane + c] = has_nw ? v.y : 0.f;
    };
    pair_equilibrium(r, u, put);
    put(0, rest);
}

dim3 brick_grid(const Geom& g) { return dim3((g.nx + MX - 1) / MX, (g.ny + MY - 1) / MY, (g.nz + MZ - 1) / MZ); }

}  // namespace

cudaError_t launch_step_moments(float* buffer, const uint32_t* nbr, const uint32_t* nbr_nw, const uint32_t* adh,
                                const Geom& g, const Phys& p, cudaStream_t s) {
    moment_gather_kernel<<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(buffer, nbr, nbr_nw, g);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    moment_collide_kernel<false><<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(buffer, nullptr, nullptr, nbr, adh, g, p);
    return cudaGetLastError();
}

cudaError_t launch_first_moments(float* F, float2* rho2, float* buffer, const uint32_t* nbr, const uint32_t* adh,
                                 const Geom& g, const Phys& p, cudaStream_t s) {
    cudaError_t e = launch_pair_moments(F, rho2, nbr, g, s);
    if (e != cudaSuccess) return e;
    moment_collide_kernel<true><<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(
        buffer, reinterpret_cast<const float2*>(F), rho2, nbr, adh, g, p);
    return cudaGetLastError();
}

cudaError_t launch_moments_to_pull(float* buffer, float* fout, const uint32_t* nbr, const Geom& g, cudaStream_t s) {
    moments_to_pull_kernel<<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(buffer, fout, nbr, g);
    return cudaGetLastError();
}

cudaError_t launch_density_moments(float* buffer, float2* rho2, float* rho, const uint32_t* nbr, const uint32_t* nbr_nw,
                                   const Geom& g, cudaStream_t s) {
    moment_density_kernel<<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(buffer, nbr, nbr_nw, g, rho2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    split_density_kernel<<<1216, 256, 0, s>>>(rho2, rho, (long long)g.nxy * g.nz);
    return cudaGetLastError();
}

cudaError_t launch_measure_moments(float* buffer, float2* rho2, const uint32_t* nbr, const uint32_t* nbr_nw,
                                   const Geom& g, double G, double* partials, int nblocks, double* result,
                                   cudaStream_t s) {
    moment_density_kernel<<<brick_grid(g), dim3(MX, MY, MZ), 0, s>>>(buffer, nbr, nbr_nw, g, rho2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    measure_density_kernel<<<nblocks, 256, 0, s>>>(rho2, nbr, (long long)g.nxy * g.nz, G, partials);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_finalize(partials, nblocks, result, s);
}

cudaError_t launch_probe_moments(float* buffer, const uint32_t* nbr, const uint32_t* nbr_nw, const Geom& g, int x,
                                 int y, int z, float* out, cudaStream_t s) {
    moment_probe_kernel<<<1, 1, 0, s>>>(buffer, nbr, nbr_nw, g, x, y, z, out);
    return cudaGetLastError();
}

}  // namespace lbmk
