// lbm_aux.cu -- per-domain set-up and read-out kernels: geometry words from the
// mask, the initial populations, the density field and the FP64 measurements.
#include "lbm_device.cuh"

namespace lbmk {

namespace {

// One thread per cell: x and y from the block and thread, z from blockIdx.z.
__global__ void __launch_bounds__(256) geometry_kernel(const uint8_t* __restrict__ mask, uint32_t* __restrict__ nbr,
                                                       uint32_t* __restrict__ nbr_nw, uint32_t* __restrict__ adh,
                                                       Geom g) {
    const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y, z = blockIdx.z;
    if (x < g.nx && y < g.ny) geometry_cell(mask, nbr, nbr_nw, adh, g, x, y, z);
}

// Stored populations whose pull yields the rest equilibrium w_k rho0(x) at every
// fluid cell: B_j(y) = w_j rho0(y + e_j) when y + e_j is fluid for the component
// (it pulls direction j from y), else w_j rho0(y) (y pulls jbar from itself).
__global__ void init_kernel(const float* __restrict__ rho0, float* __restrict__ f, const uint32_t* __restrict__ nbr,
                            const uint32_t* __restrict__ nbr_nw, Geom g) {
    const long long N = (long long)g.nxy * g.nz;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)c;  // a domain holds fewer than 2^31 cells (lbm_create_domain)
        const int x = ci % g.nx;
        const int y = (ci / g.nx) % g.ny;
        const int z = ci / g.nxy;
        const uint32_t w = nbr[c];
        const uint32_t cls = (w >> CLS_SHIFT) & CLS_MASK;
        for (int s = 0; s < 2; ++s) {
            const bool fl = cls != CLS_SOLID && !(s == 1 && cls == CLS_MEMBRANE);
            const uint32_t bits = s == 0 ? w : nbr_nw[c];
            const float* r = rho0 + (size_t)s * N;
            float* fs = f + (size_t)s * Q * g.plane;
#pragma unroll
            for (int j = 0; j < Q; ++j) {
                float v = 0.f;
                if (fl && j == 0) {
                    // rest value closes the pulled sum on rho0 exactly (sum_j w_j != 1 in FP32)
                    float sum = 0.f;
#pragma unroll
                    for (int i = 1; i < Q; ++i) sum += WK(i) * r[c];
                    v = r[c] - sum;
                } else if (fl) {
                    if ((bits >> OPP(j)) & 1u) {
                        v = WK(j) * r[c];
                    } else {
                        bool ok = true;
                        const int tx = wrap1(x + EX(j), g.nx, g.px, ok);
                        const int ty = wrap1(y + EY(j), g.ny, g.py, ok);
                        const int tz = wrap1(z + EZ(j), g.nz, g.pz, ok);
                        v = WK(j) * r[(long long)tz * g.nxy + (long long)ty * g.nx + tx];
                    }
                }
                fs[(size_t)j * g.plane + c] = v;
            }
        }
    }
}

// rho_s(x, t) = sum_k f_k(x, t) of the pulled populations (Eq. 2).
__global__ void density_kernel(const float* __restrict__ f, float* __restrict__ rho, const uint32_t* __restrict__ nbr,
                               const uint32_t* __restrict__ nbr_nw, Geom g) {
    const long long N = (long long)g.nxy * g.nz;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)c;  // a domain holds fewer than 2^31 cells (lbm_create_domain)
        const int x = ci % g.nx;
        const int y = (ci / g.nx) % g.ny;
        const int z = ci / g.nxy;
        Column col = make_column(x, y, g);
        float dummy[2][Q];
        float rw, rn;
        int cell;
        pull_cell<false>(f, nbr, nbr_nw, g, col, z, dummy, rw, rn, cell);
        rho[c] = rw;
        rho[N + c] = rn;
    }
}

constexpr int MEAS_THREADS = 256;

// Measurements of the current state (definitions in lbm.h), one FP64 partial
// per block; a second kernel adds the partials in block order.
__global__ void __launch_bounds__(MEAS_THREADS) measure_kernel(const float* __restrict__ f,
                                                               const uint32_t* __restrict__ nbr,
                                                               const uint32_t* __restrict__ nbr_nw, Geom g,
                                                               double G, double* __restrict__ partials) {
    MeasureSums sums;
    const long long N = (long long)g.nxy * g.nz;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N; c += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)c;  // a domain holds fewer than 2^31 cells (lbm_create_domain)
        const int x = ci % g.nx;
        const int y = (ci / g.nx) % g.ny;
        const int z = ci / g.nxy;
        Column col = make_column(x, y, g);
        float dummy[2][Q];
        float rw, rn;
        int cell;
        const uint32_t w = pull_cell<false>(f, nbr, nbr_nw, g, col, z, dummy, rw, rn, cell);
        sums.add((w >> CLS_SHIFT) & CLS_MASK, rw, rn, G);
    }
    sums.store<MEAS_THREADS / 32>(partials + (size_t)blockIdx.x * NMEAS);
}

// The blocks' partials added up: FIN_ROWS threads per sum, each over every
// FIN_ROWS-th block, then those in order (1216 blocks: 92 us as a single
// chain, 10 us).
constexpr int FIN_ROWS = 32;
__global__ void __launch_bounds__(FIN_ROWS* NMEAS)
    finalize_kernel(const double* __restrict__ partials, int nblocks, double* __restrict__ result) {
    __shared__ double part[FIN_ROWS][NMEAS];
    const int i = threadIdx.x % NMEAS, r = threadIdx.x / NMEAS;
    double v = 0.0;
#pragma unroll 4
    for (int b = r; b < nblocks; b += FIN_ROWS) v += partials[(size_t)b * NMEAS + i];
    part[r][i] = v;
    __syncthreads();
    if (r == 0) {
        for (int q = 1; q < FIN_ROWS; ++q) v += part[q][i];
        result[i] = v;
    }
}

int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    const long long cap = 16LL * device_sm_count();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

int device_sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    return sms;
}

cudaError_t launch_geometry(const uint8_t* mask, uint32_t* nbr, uint32_t* nbr_nw, uint32_t* adh, const Geom& g,
                            cudaStream_t s) {
    const dim3 grid((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    geometry_kernel<<<grid, dim3(32, 8), 0, s>>>(mask, nbr, nbr_nw, adh, g);
    return cudaGetLastError();
}

cudaError_t launch_init(const float* rho0, float* f, const uint32_t* nbr, const uint32_t* nbr_nw, const Geom& g,
                        cudaStream_t s) {
    const long long N = (long long)g.nxy * g.nz;
    init_kernel<<<grid_for(N, 256), 256, 0, s>>>(rho0, f, nbr, nbr_nw, g);
    return cudaGetLastError();
}

cudaError_t launch_density(const float* f, float* rho, const uint32_t* nbr, const uint32_t* nbr_nw, const Geom& g,
                           cudaStream_t s) {
    const long long N = (long long)g.nxy * g.nz;
    density_kernel<<<grid_for(N, 256), 256, 0, s>>>(f, rho, nbr, nbr_nw, g);
    return cudaGetLastError();
}

cudaError_t launch_finalize(const double* partials, int nblocks, double* result, cudaStream_t s) {
    finalize_kernel<<<1, FIN_ROWS * NMEAS, 0, s>>>(partials, nblocks, result);
    return cudaGetLastError();
}

// One cell a thread until the GPU is full: a throat-sized box is latency alone.
int measure_blocks(const Geom& g) {
    const long long N = (long long)g.nxy * g.nz;
    long long b = (N + MEAS_THREADS - 1) / MEAS_THREADS;
    const long long cap = 8LL * device_sm_count();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

cudaError_t launch_measure(const float* f, const uint32_t* nbr, const uint32_t* nbr_nw, const Geom& g, double G,
                           double* partials, int nblocks, double* result, cudaStream_t s) {
    measure_kernel<<<nblocks, MEAS_THREADS, 0, s>>>(f, nbr, nbr_nw, g, G, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_finalize(partials, nblocks, result, s);
}

}  // namespace lbmk
