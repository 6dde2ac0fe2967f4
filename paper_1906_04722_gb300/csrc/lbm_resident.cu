// lbm_resident.cu -- the throat batch's on-chip form: all steps of a pressure
// increment in one launch, a throat's populations kept in the shared memory of
// one thread-block cluster.
//
// What bounds the cell-list form is HBM: its two launches per step move about
// 470 bytes per cell update (0.51 + 0.21 ms a step for 1024 throats, 9 M cells;
// this form: 0.30 ms with the rest of the throats, 16 throats: 12 -> 5 us).  A throat has 1 to
// 30 thousand open cells of 152 bytes, so a cluster of up to 16 SMs holds it
// whole, and a step then costs instructions and shared-memory traffic only.
//
// The throat's cells (list order) are cut into one range per CTA, one cell (or
// two) per thread.  A step has two phases, a cluster barrier after each:
//   1. every thread reads its cells' 19 pairs, keeps their momenta in registers
//      and stores their densities, also into the halo of the CTAs whose cells
//      neighbour them;
//   2. every thread computes its cells' post-collision pairs (tau = 1 in both
//      components: the equilibria, which need the densities and momenta only)
//      and pushes each to the slot of the cell it streams to, in the own CTA's
//      shared memory or another's, or back into its own slots at a wall.
// No pair is read in phase 2, so one copy of the populations is enough.  All
// loads are local; what crosses CTAs is stores.
//
// With the populations on chip a step is bound by instruction issue and by the
// shared memory's 128 bytes a cycle, so an address must cost next to nothing.
// Each cell keeps, in registers, 18 packed 16-bit byte offsets of its
// neighbours' densities (own range, halo, or a zero entry where the neighbour
// is no fluid): an offset is used as it is for the density and, with a constant
// added, for the push, and one bit a direction says "wall" or "another CTA's".
#include <atomic>

#include "lbm_collide_pair.cuh"
#include "lbm_resident.h"

namespace lbmk {

namespace {

__device__ __forceinline__ uint32_t cluster_address(uint32_t local, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
// v to the own CTA's address `local`, or (remote != 0) to the cluster address:
// one of two predicated stores, no branch.
__device__ __forceinline__ void push_store(uint32_t remote, uint32_t local, uint32_t far, float2 v) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %0, 0;\n @!p st.shared.v2.f32 [%1], {%3, %4};\n"
        " @p st.shared::cluster.v2.f32 [%2], {%3, %4};\n}\n" ::"r"(remote),
        "r"(local), "r"(far), "f"(v.x), "f"(v.y)
        : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
    cluster_arrive();
    cluster_wait();
}
// List order is memory order: a neighbour of direction k that another CTA holds
// is the next one's when e_k points towards later cells, else the one's before.
__host__ __device__ constexpr bool points_on(int k) { return EZ(k) ? EZ(k) > 0 : EY(k) ? EY(k) > 0 : EX(k) > 0; }

// Shared memory of a CTA of S cells with halos of HM cells, in pairs: densities
// [HM | S | HM], a zero entry, then the moving populations [Q - 1][S] (the rest
// pair, which never leaves its cell, stays in registers).
template <int S, int HM>
struct Smem {
    static constexpr int ZERO = S + 2 * HM;
    static constexpr int A = ZERO + 1;
    static constexpr int PAIRS = A + (Q - 1) * S;
    static_assert(8 * ZERO < 65536, "offsets are 16 bits");
};

template <int T, int CPT, int HM, int MINB>
__global__ void __launch_bounds__(T, MINB)
    resident_kernel(const ResidentThroat* __restrict__ list, const float2* fin, float2* fout, int cp,
                    const uint32_t* __restrict__ wc, const uint32_t* __restrict__ adhc,
                    const uint4* __restrict__ rows, Phys P, const float* __restrict__ bc_all, int ladder_stride,
                    const int* __restrict__ incr_now, int n_steps) {
    constexpr int S = T * CPT;  // cells a CTA holds
    using M = Smem<S, HM>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    // offsets below are those of a cell's density: pair (HM + cell); slot k of its
    // populations (k >= 1) is POP + k * 8 S further
    constexpr int POP = 8 * (M::A - HM - S);
    auto at = [&](uint32_t off) -> float2& { return *reinterpret_cast<float2*>(smem_raw + off); };
    int rank, C;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
    const ResidentThroat th = list[blockIdx.x / C];
    const int H = th.reach;
    // cells per CTA: at least the reach, so that a neighbour is this CTA's, the one
    // before's or the one after's (the last CTAs of a small throat hold none)
    const int per = max((th.n + C - 1) / C, H), r0 = rank * per;
    const int cnt = max(0, min(per, th.n - r0));
    const uint32_t per8 = 8u * (uint32_t)per;
    const float* bc = bc_all + 4 * ((size_t)th.id * ladder_stride + *incr_now);
    if (threadIdx.x == 0) at(8 * M::ZERO) = make_float2(0.f, 0.f);

    // constant per cell: packed neighbour offsets; direction bits "wall" (bits 1
    // .. 18) with the cell's class (bits 19 .. 21), direction bits "another
    // CTA's", adhesion word
    uint32_t nb[CPT][9] = {}, wall[CPT] = {}, remote[CPT] = {}, ad[CPT] = {};
    float2 rest[CPT] = {};
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int i = (int)threadIdx.x + c * T;
        if (i >= cnt) continue;
        const int item = th.item0 + r0 + i;
        const uint32_t w = wc[item];
        ad[c] = (w & BIT_ADH) ? adhc[item] : 0u;
        const uint4 q = rows[item];
        const uint32_t row[4] = {q.x, q.y, q.z, q.w};
        wall[c] = w & (CLS_MASK << CLS_SHIFT);
#pragma unroll
        for (int k = 1; k < Q; ++k) {
            int t;  // item of x + e_k, relative to the CTA's first
            if (EY(k) == 0 && EZ(k) == 0) {
                t = i + EX(k);
            } else {
                const int r = resident_row(EY(k), EZ(k));
                t = (int)((row[r >> 1] >> (16 * (r & 1))) & 0xffffu) - r0;
                if (EX(k) < 0) t -= 1;
                // the row's cell at x itself precedes x + 1 where it is open
                if (EX(k) > 0) t += 1 - (int)((w >> OPP(resident_row_dir(EY(k), EZ(k)))) & 1u);
            }
            uint32_t off = 8u * (uint32_t)(HM + t);
            if ((w >> OPP(k)) & 1u) {
                wall[c] |= 1u << k;
                off = 8u * M::ZERO;
            } else if ((unsigned)t >= (unsigned)per) {
                remote[c] |= 1u << k;
            }
            nb[c][(k - 1) >> 1] |= off << (16 * ((k - 1) & 1));
        }
        const uint32_t self = 8u * (uint32_t)(HM + i);
        rest[c] = fin[item];
#pragma unroll
        for (int k = 1; k < Q; ++k) at(self + POP + 8 * S * k) = fin[(size_t)k * cp + item];
    }
    auto offset = [&](int c, int k) -> uint32_t {
        return ((k - 1) & 1) ? nb[c][(k - 1) >> 1] >> 16 : nb[c][(k - 1) >> 1] & 0xffffu;
    };
    // cluster addresses of offset 0 in the CTAs before and after, moved so that an
    // offset of this CTA's range lands on the same item there
    const uint32_t before = cluster_address(smem0, max(rank - 1, 0)) + per8;
    const uint32_t after = cluster_address(smem0, min(rank + 1, C - 1)) - per8;
    cluster_barrier();  // every CTA of the cluster has started: its shared memory may be written

    for (int step = 0; step < n_steps; ++step) {
        // unpacked offsets are not worth a register across steps: hide from the
        // compiler that the packed ones stay the same
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
#pragma unroll
            for (int r = 0; r < 9; ++r) asm volatile("" : "+r"(nb[c][r]));
            asm volatile("" : "+r"(wall[c]), "+r"(remote[c]), "+r"(ad[c]));
        }
        float2 j[CPT][3];
        float up[CPT][3];
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
            const int i = (int)threadIdx.x + c * T;
            if (i >= cnt) continue;
            const uint32_t self = 8u * (uint32_t)(HM + i);
            float2 r;
            pair_moments([&](int k) { return k ? at(self + POP + 8 * S * k) : rest[c]; }, r, j[c]);
            at(self) = r;
            if (i < H && rank > 0) cluster_store(before + self, r);
            if (i >= per - H && rank + 1 < C) cluster_store(after + self, r);
        }
        cluster_arrive();
#pragma unroll
        for (int c = 0; c < CPT; ++c) {  // while the densities travel: what needs none of them
            const int i = (int)threadIdx.x + c * T;
            if (i < cnt) pair_common_velocity(at(8u * (uint32_t)(HM + i)), j[c], up[c]);
        }
        cluster_wait();
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
            const int i = (int)threadIdx.x + c * T;
            if (i >= cnt) continue;
            const uint32_t self = 8u * (uint32_t)(HM + i);
            const uint32_t cls = (wall[c] >> CLS_SHIFT) & CLS_MASK;
            float2 r = at(self), u[3];
            const bool open_end = cls == CLS_INLET || cls == CLS_OUTLET;
            if (open_end) {
                const float* b = bc + (cls == CLS_INLET ? 0 : 2);
                r = make_float2(__ldg(b), __ldg(b + 1));
                u[0] = u[1] = u[2] = pair2(0.f);
            } else {
                pair_velocity(r, up[c], ad[c], P, [&](int k) { return at(offset(c, k)); }, u);
            }
            rest[c] = pair_equilibrium(r, u, [&](int k, float2 v) {
                const uint32_t o = offset(c, k), slot = POP + 8 * S * k;
                // a wall sends the value back into the opposite slot (k + 1 or k - 1)
                const uint32_t back = OPP(k) > k ? self + 8 * S : self - 8 * S;
                push_store(remote[c] & (1u << k), smem0 + (wall[c] & (1u << k) ? back : o) + slot,
                           (points_on(k) ? after : before) + o + slot, v);
            });
            if (open_end) rest[c] = pair_reservoir_rest(r);
        }
        cluster_barrier();
    }
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const int i = (int)threadIdx.x + c * T;
        if (i >= cnt) continue;
        const int item = th.item0 + r0 + i;
        const uint32_t self = 8u * (uint32_t)(HM + i);
        fout[item] = rest[c];
#pragma unroll
        for (int k = 1; k < Q; ++k) fout[(size_t)k * cp + item] = at(self + POP + 8 * S * k);
    }
}

// A CTA of 1024 threads and one cell each has the shorter step; 704 threads of
// two cells hold the larger throats, and any throat on fewer SMs.
struct Shape {
    int threads, cells, halo;
    size_t smem;
};
constexpr int HALO0 = 1536, HALO1 = 1150;
constexpr Shape SHAPES[RESIDENT_SHAPES] = {{1024, 1024, HALO0, sizeof(float2) * Smem<1024, HALO0>::PAIRS},
                                           {704, 1408, HALO1, sizeof(float2) * Smem<1408, HALO1>::PAIRS}};
static_assert(SHAPES[0].smem <= RESIDENT_SMEM && SHAPES[1].smem <= RESIDENT_SMEM, "shared memory");

using Kernel = void (*)(const ResidentThroat*, const float2*, float2*, int, const uint32_t*, const uint32_t*,
                        const uint4*, Phys, const float*, int, const int*, int);
Kernel kernel_of(int shape) {
    return shape == 0 ? resident_kernel<1024, 1, HALO0, 1> : resident_kernel<704, 2, HALO1, 1>;
}

cudaLaunchConfig_t launch_config(int shape, int cluster, int n_throats, cudaLaunchAttribute (&attr)[2],
                                 cudaStream_t s) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_throats * cluster));
    cfg.blockDim = dim3((unsigned)SHAPES[shape].threads);
    cfg.dynamicSmemBytes = SHAPES[shape].smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Row positions of the items [first, n): eight 16-bit positions in the throat's
// own list (the table of resident_kernel); the entry of a solid cell at x is
// the position an item there would have.
__global__ void __launch_bounds__(256)
    resident_rows_kernel(const int2* __restrict__ items, int first, int n,
                         const ResidentBox* __restrict__ boxes, const int* __restrict__ box_to_item,
                         const uint32_t* __restrict__ nbr, const uint32_t* __restrict__ adh, uint32_t* __restrict__ wc,
                         uint32_t* __restrict__ adhc, uint4* __restrict__ rows) {
    const int i = first + blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int2 it = items[i];
    const ResidentBox g = boxes[it.x];
    const int x = it.y & 1023, y = (it.y >> 10) & 1023, z = it.y >> 20;
    const long long cell = g.c_off + ((long long)z * g.ny + y) * g.nx + x;
    const uint32_t w = nbr[cell];
    wc[i] = w;
    adhc[i] = (w & BIT_ADH) ? adh[cell] : 0u;
    const int item0 = g.item0;
    auto at = [&](int dy, int dz) -> uint32_t {
        const int yy = y + dy, zz = z + dz;
        if (yy < 0 || yy >= g.ny || zz < 0 || zz >= g.nz) return 0u;
        const int* m = box_to_item + g.c_off + ((long long)zz * g.ny + yy) * g.nx + x;
        if (m[0] >= 0) return (uint32_t)(m[0] - item0);
        if (x + 1 < g.nx && m[1] >= 0) return (uint32_t)(m[1] - item0);
        if (x > 0 && m[-1] >= 0) return (uint32_t)(m[-1] + 1 - item0);
        return 0u;
    };
    // in the order of resident_row
    rows[i - first] = make_uint4(at(1, 0) | at(-1, 0) << 16, at(0, 1) | at(0, -1) << 16, at(1, 1) | at(-1, -1) << 16,
                         at(1, -1) | at(-1, 1) << 16);
}

}  // namespace

int resident_cells(int shape) { return SHAPES[shape].cells; }

int resident_max_reach(int shape) { return SHAPES[shape].halo; }

int resident_clusters(int shape, int cluster) {
    // what the device holds does not change: asked once per device
    constexpr int DEVICES = 64;
    static std::atomic<int> known[DEVICES][RESIDENT_SHAPES][RESIDENT_MAX_CLUSTER + 1];  // held + 1, 0: not asked
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::atomic<int>* seen = dev >= 0 && dev < DEVICES ? &known[dev][shape][cluster] : nullptr;
    if (seen && seen->load() > 0) return seen->load() - 1;
    const void* k = reinterpret_cast<const void*>(kernel_of(shape));
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config(shape, cluster, 1, attr, nullptr);
    int held = 0;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SHAPES[shape].smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&held, k, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();  // not a failure of the caller's: the throat goes another way
        return 0;
    }
    if (seen) seen->store(held + 1);
    return held;
}

cudaError_t launch_resident(int shape, int cluster, int n_throats, const ResidentThroat* list, const float2* fin,
                            float2* fout, int cp, const uint32_t* wc, const uint32_t* adhc, const uint4* rows,
                            const Phys& P, const float* bc, int ladder_stride, const int* incr, int n_steps,
                            int rank, cudaStream_t s) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = launch_config(shape, cluster, n_throats, attr, s);
    // launches side by side: the lower the rank the sooner its clusters are placed
    int least = 0, greatest = 0;
    if (cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest); e != cudaSuccess) return e;
    attr[1].id = cudaLaunchAttributePriority;
    attr[1].val.priority = greatest + rank < least ? greatest + rank : least;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel_of(shape), list, fin, fout, cp, wc, adhc, rows, P, bc, ladder_stride, incr,
                              n_steps);
}

cudaError_t launch_resident_rows(const int2* items, int first, int n, const ResidentBox* boxes, const int* box_to_item,
                                 const uint32_t* nbr, const uint32_t* adh, uint32_t* wc, uint32_t* adhc, uint4* rows,
                                 cudaStream_t s) {
    if (n <= first) return cudaSuccess;
    resident_rows_kernel<<<(unsigned)((n - first + 255) / 256), 256, 0, s>>>(items, first, n, boxes,
                                                                             box_to_item, nbr, adh, wc, adhc, rows);
    return cudaGetLastError();
}

}  // namespace lbmk
