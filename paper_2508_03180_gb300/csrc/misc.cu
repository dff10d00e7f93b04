// Layout conversion between the ABI's per-parameter row-major arrays and the
// library's structure-of-arrays planes, and the L1 photometric loss.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "internal.cuh"

namespace dgs {

// Row-major arrays src [rows][cols] into planes: column c at dst + c * stride.
// One launch takes all arrays of a scene in tiles of about PL_ELEMS elements
// (a whole number of 32-row groups), so that every array keeps the
// same bytes in flight whatever its width and a small scene pays for one launch:
// the tile's rows are read as one contiguous run, sixteen bytes a thread where
// the array is aligned, turned in shared memory (odd row stride: no bank conflicts) and
// written as runs of consecutive rows per plane.  Bound by HBM: the five arrays of
// 1M Gaussians at SH 3 (472 MB read and written) took 220 us in five launches of
// 32-row blocks, 148 us this way with divisions in the index arithmetic and 130 without.
constexpr int PL_T = 256, PL_ELEMS = 4096;
__global__ void __launch_bounds__(PL_T) k_rows_to_planes(const PlaneCopies C) {
    __shared__ __align__(16) float t[PL_ELEMS + PL_ELEMS / 2];  // rows x (cols | 1): widest for two columns
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int64_t task = blockIdx.x; task < C.tasks; task += gridDim.x) {
        int a = 0;
        while (a + 1 < C.n && C.a[a + 1].first_task <= task) ++a;
        const PlaneCopy &P = C.a[a];
        const int cols = P.cols, ld = cols | 1, tr = plane_tile_rows(cols);
        const int64_t r0 = (task - P.first_task) * tr;
        const int nr = (int)min((int64_t)tr, P.rows - r0), ne = nr * cols;
        const float *src = P.src + r0 * cols;
        const uint32_t magic = cols > 1 ? (uint32_t)(((1ull << 32) + cols - 1) / cols) : 0u;
        // i / cols by the exact reciprocal (i, cols < 2^16); element i belongs at i, or with
        // an even row length (and the odd stride) at i + row
        auto row = [&](uint32_t i) { return cols > 1 ? __umulhi(i, magic) : i; };
        const int n4 = ((uintptr_t)P.src & 15) == 0 ? ne / 4 : 0;  // (r0 * cols is a multiple of 32)
        if (cols & 1) {
#pragma unroll 4
            for (int i = tid; i < n4; i += PL_T) reinterpret_cast<float4 *>(t)[i] = reinterpret_cast<const float4 *>(src)[i];
            for (int i = 4 * n4 + tid; i < ne; i += PL_T) t[i] = src[i];
        } else {
#pragma unroll 4
            for (int i = tid; i < n4; i += PL_T) {
                const float4 v = reinterpret_cast<const float4 *>(src)[i];
                t[4 * i + row(4 * i)] = v.x;
                t[4 * i + 1 + row(4 * i + 1)] = v.y;
                t[4 * i + 2 + row(4 * i + 2)] = v.z;
                t[4 * i + 3 + row(4 * i + 3)] = v.w;
            }
            for (int i = 4 * n4 + tid; i < ne; i += PL_T) t[i + row(i)] = src[i];
        }
        __syncthreads();
        // warp w: 32-row groups of the planes, group-major
        const int groups = (nr + 31) / 32;
#pragma unroll 4
        for (int u = warp; u < groups * cols; u += PL_T / 32) {
            const int g = (int)row(u), c = u - g * cols, r = 32 * g + lane;
            if (r < nr) P.dst[c * P.stride + r0 + r] = t[r * ld + c];
        }
        __syncthreads();
    }
}

__global__ void k_soa_to_aos(const float *__restrict__ src, int64_t rows, int cols, int64_t src_stride,
                             float *__restrict__ dst) {
    const int64_t total = rows * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / cols;
        const int c = (int)(i - r * cols);
        dst[i] = src[c * src_stride + r];
    }
}

__global__ void k_fill(float *__restrict__ dst, int64_t n, float v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = v;
}

long long resident_ctas(const void *kernel, int threads) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, long long> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(dev, kernel);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int sms = 0, per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev < 0 ? 0 : dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    const long long n = (long long)std::max(1, sms) * std::max(1, per_sm);
    cache[key] = n;
    return n;
}

static int grid_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

void PlaneCopies::add(const float *src, int64_t rows, int cols, float *dst, int64_t stride) {
    if (rows * cols == 0) return;
    if (rows == 1 && stride == 1) { rows = cols; cols = 1; }  // one row: a plain copy
    a[n++] = PlaneCopy{src, dst, rows, stride, tasks, cols};
    const int tr = plane_tile_rows(cols);
    tasks += (rows + tr - 1) / tr;
}

void launch_rows_to_planes(const PlaneCopies &c, cudaStream_t st) {
    if (c.tasks == 0) return;
    k_rows_to_planes<<<(unsigned)std::min<int64_t>(c.tasks, 152 * 8), PL_T, 0, st>>>(c);
}

void launch_soa_to_aos(const float *src, int64_t rows, int cols, int64_t src_stride, float *dst, cudaStream_t st) {
    if (rows * cols == 0) return;
    k_soa_to_aos<<<grid_for(rows * cols), 256, 0, st>>>(src, rows, cols, src_stride, dst);
}

void launch_fill_f32(float *dst, int64_t n, float v, cudaStream_t st) {
    if (n == 0) return;
    k_fill<<<grid_for(n), 256, 0, st>>>(dst, n, v);
}

// L1 loss: dL/drgb = sign(rgb - target) / n; per-block partial sums of
// |rgb - target| then a single-block sum in fixed order (deterministic).
constexpr int LOSS_T = 256;

int loss_l1_blocks(int64_t n) {
    int64_t b = (n + LOSS_T * 8 - 1) / (LOSS_T * 8);
    if (b > 152 * 8) b = 152 * 8;
    return (int)(b < 1 ? 1 : b);
}

__device__ __forceinline__ float block_sum(float v, float *s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < LOSS_T / 32; ++w) t += s[w];
    return t;
}

__global__ void __launch_bounds__(LOSS_T) k_loss_l1(const float *__restrict__ rgb, const float *__restrict__ target,
                                                    int64_t n, float inv_n, float *__restrict__ dL,
                                                    float *__restrict__ partial) {
    __shared__ float s[LOSS_T / 32];
    float acc = 0.f;
    for (int64_t i = blockIdx.x * (int64_t)LOSS_T + threadIdx.x; i < n; i += (int64_t)gridDim.x * LOSS_T) {
        const float d = rgb[i] - target[i];
        acc += fabsf(d);
        dL[i] = d > 0.f ? inv_n : (d < 0.f ? -inv_n : 0.f);
    }
    const float t = block_sum(acc, s);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void __launch_bounds__(LOSS_T) k_loss_final(const float *__restrict__ partial, int nb, float inv_n,
                                                       float *__restrict__ loss) {
    chain_wait();
    __shared__ float s[LOSS_T / 32];
    float acc = 0.f;
    for (int i = threadIdx.x; i < nb; i += LOSS_T) acc += partial[i];
    const float t = block_sum(acc, s);
    if (threadIdx.x == 0) *loss = t * inv_n;
}

void launch_loss_l1(const float *rgb, const float *target, int64_t n, float *dL, float *partial, int nblocks,
                    float *loss, cudaStream_t st) {
    const float inv_n = n > 0 ? 1.0f / (float)n : 0.f;
    k_loss_l1<<<nblocks, LOSS_T, 0, st>>>(rgb, target, n, inv_n, dL, partial);
    launch_chained(k_loss_final, 1, LOSS_T, 0, st, partial, nblocks, inv_n, loss);
}

}  // namespace dgs
