// lbm_resident.h -- the throat batch's on-chip form (lbm_resident.cu): a
// throat's populations in the shared memory of one thread-block cluster for all
// steps of an increment.
#pragma once

#include "lbm_internal.h"

namespace lbmk {

constexpr int RESIDENT_SHAPES = 2;
constexpr int RESIDENT_MAX_CLUSTER = 16;
constexpr size_t RESIDENT_SMEM = 232448;  // shared memory a CTA may use (227 KB)

// Rows of neighbours (ey, ez) in the order of the row positions, and the
// direction of a row's cell at the same x.
__host__ __device__ constexpr int resident_row(int ey, int ez) {
    return ez == 0 ? (ey > 0 ? 0 : 1) : ey == 0 ? (ez > 0 ? 2 : 3) : ey > 0 ? (ez > 0 ? 4 : 6) : (ez < 0 ? 5 : 7);
}
__host__ __device__ constexpr int resident_row_dir(int ey, int ez) {
    for (int k = 1; k < Q; ++k)
        if (EX(k) == 0 && EY(k) == ey && EZ(k) == ez) return k;
    return 0;
}

// One throat: its items [item0, item0 + n) of the list, its index in the batch,
// and the largest distance in the list between an item and a neighbour.
struct ResidentThroat {
    int item0, n, reach, id;
};
// Box of a throat for the position table.
struct ResidentBox {
    long long c_off;
    int nx, ny, nz, item0;
};

int resident_cells(int shape);      // cells a CTA of the shape holds
int resident_max_reach(int shape);  // largest reach the shape has room for
// Clusters of this size that the current device holds at once (0: the kernel
// cannot be launched that way).
int resident_clusters(int shape, int cluster);
// n_steps time steps of n_throats throats (cluster CTAs each): pairs from fin
// into fout (which may be the same array), strides cp.  A throat's reach must not
// exceed resident_max_reach, and max(n / cluster, reach) not resident_cells.  rank: 0 for the first of
// several launches that run side by side.
cudaError_t launch_resident(int shape, int cluster, int n_throats, const ResidentThroat* list, const float2* fin,
                            float2* fout, int cp, const uint32_t* wc, const uint32_t* adhc, const uint4* rows,
                            const Phys& P, const float* bc, int ladder_stride, const int* incr, int n_steps,
                            int rank, cudaStream_t s);
// Geometry and adhesion words of the items [first, n) (at their own index) and
// their row positions (rows[0] is item first's).
cudaError_t launch_resident_rows(const int2* items, int first, int n, const ResidentBox* boxes, const int* box_to_item,
                                 const uint32_t* nbr, const uint32_t* adh, uint32_t* wc, uint32_t* adhc, uint4* rows,
                                 cudaStream_t s);

}  // namespace lbmk
