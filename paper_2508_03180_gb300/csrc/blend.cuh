// Helpers shared by the blend kernels: the hybrid's (blend.cu) and the comparators'
// (compare.cu).  One warp per 16x8 sub-tile of a tile, four pixels per lane,
// the tile's list taken in batches of 32 records staged in shared memory.
#pragma once
#include "internal.cuh"

namespace dgs {

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int find_view(const ViewDesc *views, int n_views, int tile) {
    int lo = 0, hi = n_views;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (views[mid].tile_base <= tile) lo = mid; else hi = mid;
    }
    return lo;
}

// Can record piece r0 pass the AABB test at some pixel centre of the 16-wide,
// `rows`-high block whose first pixel is (x0, y0)?  Exactly conservative (FP32
// subtraction is monotone, so testing the nearest pixel centres suffices).
__device__ __forceinline__ bool touches_rows(float4 r0, float x0, float y0, float rows) {
    const float lx = x0 + 0.5f, hx = x0 + (float)kTile - 0.5f;
    const float ly = y0 + 0.5f, hy = y0 + rows - 0.5f;
    return !(lx - r0.x > r0.z || r0.x - hx > r0.z || ly - r0.y > r0.w || r0.y - hy > r0.w);
}

// Does record piece r0 pass the AABB test at every pixel centre of the block?
// Exact: testing its first and last columns and rows suffices (FP32
// subtraction is monotone, so every offset lies between theirs).
__device__ __forceinline__ bool covers_rows(float4 r0, float x0, float y0, float rows) {
    const float lx = x0 + 0.5f, hx = x0 + (float)kTile - 0.5f;
    const float ly = y0 + 0.5f, hy = y0 + rows - 0.5f;
    return fabsf(lx - r0.x) <= r0.z && fabsf(hx - r0.x) <= r0.z && fabsf(ly - r0.y) <= r0.w &&
           fabsf(hy - r0.y) <= r0.w;
}

// Pixels of a lane in a 16 x (2 PPL) sub-tile: lane l = 8 j + i takes the
// columns i and i + 8 and the rows j + 4 r (r < PPL / 2); pixel q = 2 r + c.
// Each q thus spans an 8x4 quadrant of the warp's lanes, which meets fewer
// (quadrant, Gaussian) pairs than a 16x2 strip: a Gaussian's AABB is about
// square, and the per-pixel work of a quadrant runs whenever any of its
// pixels is hit (17% fewer such runs than one column per lane on the
// benchmark scene).
__device__ __forceinline__ int lane_col(int lane, int c) { return (lane & 7) + 8 * c; }
__device__ __forceinline__ int lane_row(int lane, int r) { return (lane >> 3) + 4 * r; }

// Cells of a tile list in batches: the 32 / K cells (one at least) whose Gaussians a
// warp's lanes test in one ballot.  Lane l copies the float4s l, l + 32, l + 64
// of a batch (at most 32 records), whose cell within the batch and place within the
// cell stay the same for the whole list; the ids of a batch's cells are read one
// batch before its copies are issued, so no copy waits for its address.
constexpr int FSTAGE = 2;          // batches in shared memory: one blended, one on its way
constexpr int kBatchF4 = 32 * kRecF4;
__host__ __device__ constexpr int batch_cells(int K) { return 32 / K; }

struct CellBatches {
    const uint32_t *__restrict__ cells;
    const float4 *__restrict__ vrec;
    uint32_t end;
    uint32_t id;            // lane l: cell l of the next batch to copy
    uint32_t pos;           // byte q: the cell (of the batch) of the lane's q-th piece
    __device__ __forceinline__ CellBatches(const uint32_t *c, const float4 *v, uint32_t list_end, int K, int lane)
        : cells(c), vrec(v + lane), end(list_end), id(0u), pos(0u) {
#pragma unroll
        for (int q = 0; q < 3; ++q) pos |= (uint32_t)((lane + 32 * q) / (kRecF4 * K)) << (8 * q);
    }
    // cells of the batch at entry e
    __device__ __forceinline__ uint32_t count(uint32_t e, int K) const {
        return e < end ? min(end - e, (uint32_t)batch_cells(K)) : 0u;
    }
    __device__ __forceinline__ void read_ids(uint32_t e, int K, int lane) {
        if (lane < count(e, K)) id = __ldg(cells + e + lane);
    }
    // the copies of the batch at entry e (its ids read before)
    __device__ __forceinline__ void issue(float4 *dst, uint32_t e, int K, int lane) const {
        const uint32_t n = count(e, K);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const uint32_t j = (pos >> (8 * q)) & 255u, from = __shfl_sync(0xffffffffu, id, j);
            // piece lane + 32 q of the batch is piece lane + 32 q - j per of its cell
            if (j < n) cp_async16(dst + lane + 32 * q, vrec + ((long long)from - j) * (kRecF4 * K) + 32 * q);
        }
    }
};

}  // namespace dgs
