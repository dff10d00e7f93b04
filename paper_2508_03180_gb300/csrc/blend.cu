// Physical weighted-sum blend (Layer II, Sec. V) and its adjoint.
//
// Per pixel, the tile's cells are walked front to back (the order of the
// cell sort).  For cell n with Gaussians k:
//     A_n = sum_k alpha_k c_k,  B_n = sum_k alpha_k,  P_n = prod_k (1 - v_n alpha_k)
//     N += v_n T_n A_n,  D += v_n T_n B_n,  T_{n+1} = T_n P_n          (Eq. 12-14)
// and the pixel is C = N / D.  Before cell n the pixel stops if T_n < eps
// (cell-level early termination, Sec. V-B).  alpha_k = min(sigma G'(x'),
// alpha_max) and is 0 when the pixel lies outside the Gaussian's AABB
// (false-positive skip, Sec. VI-A).  Inside a cell nothing depends on the
// order of k (Eq. 12's inner sums and product commute).
//
// GB300 mapping: one one-warp CTA per 16x8 half of a 16x16 tile, four
// pixels per lane in packed pairs (f32x2 arithmetic), or per 16x4 quarter, two
// pixels per lane, where there are few tiles (kFewTiles).  The 48-byte records of
// the cells' Gaussians are copied into the warp's shared memory asynchronously,
// ahead of their use, and broadcast from there to the warp's 128 pixels.
#include <algorithm>
#include <type_traits>

#include "blend.cuh"

namespace dgs {

constexpr int BT = 256;
constexpr float LN2 = 0.6931471805599453f;

// Work unit: one warp (a one-warp CTA) per 16 x (2 PPL)-pixel sub-tile of a
// tile.  Warps never wait for one another: each stages the records of its
// tile's cells in its own shared memory, takes a ballot of a cell's Gaussians
// whose AABB reaches its sub-tile and loops over those only, and stops as soon
// as its own pixels are done.  KT > 0 fixes K at compile time.
constexpr int WT = 32;  // threads per work unit

// The adjoint's records reach shared memory by asynchronous copies (cp.async, 16 bytes
// a lane, one to three per lane for a cell), three cells deep: the copy of
// entry e + 2 is issued while entry e is blended, so neither registers nor a
// wait on the load's latency are spent on staging.  Every iteration commits one
// copy group (empty past the list's end) and waits for all but the two
// newest, which are the next two entries' (cp_async16 and friends: internal.cuh).
// (The forward takes its cells in batches: CellBatches.  In the adjoint batches
// were no faster, 5.16 -> 5.19 ms with one buffer and 5.28 with two.)
constexpr int NSTAGE = 3;

// Issue the copy of the records of cell `id` (per float4s) into dst.
// KT > 0: K at compile time (one or two pieces a lane for the common ones).
template <int KT>
__device__ __forceinline__ void issue_cell(float4 *dst, const float4 *__restrict__ vrec, uint32_t id, int per,
                                           int lane) {
    const float4 *src = vrec + (long long)id * per;
    constexpr int PIECES = ((KT > 0 ? KT : kMaxK) * kRecF4 + 31) / 32;
#pragma unroll
    for (int q = 0; q < PIECES; ++q) {
        const int i = lane + 32 * q;
        if (i < per) cp_async16(dst + i, src + i);
    }
}

// Cell ids of a tile list, read 32 at a time (lane j holds entry base + j)
// and handed out by a shuffle; entries must be asked for in increasing order
// from `first`, one at a time.
struct CellFeed {
    const uint32_t *__restrict__ cells;
    uint32_t first, end, chunk;
    __device__ __forceinline__ uint32_t id(uint32_t e, int lane) {
        const int j = (int)((e - first) & 31u);
        if (j == 0) chunk = e + lane < end ? __ldg(cells + e + lane) : 0u;
        return __shfl_sync(0xffffffffu, chunk, j);
    }
};

// The forward's work unit: one warp per 16 x (2 PPL) sub-tile.  FWD_PPL = 4
// (16x8 sub-tiles, the adjoint's): with the pixel math in packed pairs, the
// per-Gaussian work of a lane (record loads, AABB tests) spread over four
// pixels outweighs the register cost; the kernels are held to 64 registers
// (32 one-warp CTAs per SM).
//
// Bound by instruction issue.  A (sub-tile, cell) pair has two Gaussians in reach
// on average, about 90 of the 200 warp instructions that a cell cost when it was
// copied, tested and added up by itself: a batch's copies, wait and ballots now
// serve 32 / K cells, and a cell with no Gaussian in reach (P = 1, sums 0) leaves
// the pixels as they are and costs nothing more.  1M Gaussians, eight 1080p views:
// 2.16 -> 1.97 ms; two views of neural cells, fewer hits per cell: 0.65 -> 0.52 ms;
// 2,048 cells x 8 at 256 x 256, one warp a scheduler: 74 -> 46 us.  Weighting every
// alpha by v_n T_n instead of the cell's sums (no sums to clear and add) takes
// another 3%, but rounds N and D more often; 72 registers and 28 CTAs an SM: 2.00 ms.
// Of 74 instructions per visited Gaussian then left, the minimum with alpha_max is
// needed only where an opacity reaches it (a batch without one takes a copy of the
// loop that has none), and offsets and row squares are formed in pairs: 1.95 -> 1.85 ms.
// (In the adjoint's first pass neither pays: 5.10 -> 5.11 and 5.21 ms.)
constexpr int FWD_PPL = 4;
// an offset from the Gaussian's centre that no box reaches: s1 or s2 then
// squares to at least ~1e18 (the record's L entries are far above 1e-9), and
// exp2 of its negation is +0
constexpr float kFar = 1e18f;
constexpr int FWD_SUB = kTile / (2 * FWD_PPL);  // sub-tiles per tile
// Up to this many tiles the kernels take 16x4 sub-tiles (two pixels per lane) instead:
// with fewer than eight 16x8 warps a scheduler, a view takes as long as its longest
// list's chain of latencies, and the smaller sub-tile's list has fewer Gaussians in
// reach (one view, 16x8 / 16x4, us: forward 256x256 of 2,048 x 8 46 / 31, 320x240 of
// 20,000 x 8 141 / 88, 640x480 of 20,000 x 10 over three decades 71 / 59, 1024x576 of
// 12,345 x 7 92 / 76; adjoint 124 / 79, 376 / 228, 185 / 145, and 960x540 186 / 159); at
// 3,600 tiles its extra instructions count (1280x720 of 60,000 x 10: 163 / 182 and
// 402 / 466; 20,011 x 5, 3,690 tiles: equal, and 353 / 360).  Per pixel both do the same
// operations in the same order.
constexpr int kFewTiles = 2304;
constexpr int fwd_minb(bool var) { return var ? 24 : 32; }  // (the variants spill at 64 registers)

// VAR: the variant flags and background weight are live (dgs_config.flags,
// w_bg); without it the kernels are the paper's reading with no check left.
template <int KT, int PPL, bool VAR>
__device__ __forceinline__ void blend_fwd_unit(int unit, const ViewDesc *__restrict__ views, int n_views,
                                               const uint32_t *__restrict__ order,
                                               const uint2 *__restrict__ ranges, const uint32_t *__restrict__ cells,
                                               const float4 *__restrict__ rec, const BlendParams &bp,
                                               float *__restrict__ out_rgb, float *__restrict__ out_rgb2,
                                               float *__restrict__ out_D, int *__restrict__ out_nd,
                                               float4 (*s_rec)[kBatchF4]) {
    constexpr int ROWS = 2 * PPL, NSUB = kTile / ROWS;
    const int lane = threadIdx.x;
    const int tile = (int)order[unit / NSUB], sub = unit % NSUB;
    const int vi = find_view(views, n_views, tile);
    const ViewDesc &V = views[vi];
    const int local = tile - V.tile_base;
    const int tx = local % V.Tx, ty = local / V.Tx;
    const float bx0 = (float)(tx * kTile), by0 = (float)(ty * kTile + ROWS * sub);
    constexpr int NR = PPL / 2;  // rows per lane
    int xs[2], ys[NR];
    float pxs[2], pys[NR];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        xs[c] = tx * kTile + lane_col(lane, c);
        pxs[c] = (float)xs[c] + 0.5f;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        ys[r] = ty * kTile + ROWS * sub + lane_row(lane, r);
        pys[r] = (float)ys[r] + 0.5f;
    }
    const int K = KT > 0 ? KT : V.K;
    const uint32_t CB = batch_cells(K);
    const unsigned kmask = K == 32 ? 0xffffffffu : (1u << K) - 1u;
    const unsigned kinv = (65535u + (unsigned)K) / (unsigned)K;  // l / K = l kinv >> 16 for l < 32
    const uint2 rg = ranges[tile];

    // A pixel is done once T < eps (eps >= 0): T is then not needed any more and holds,
    // as a negative number, how many cells were blended (done_after).
    // A lane's two pixels of a row as packed pairs (one f32x2 operation per pair;
    // per component the same IEEE operations as one pixel).
    float T[PPL];
    float2 N0[NR], N1[NR], N2[NR], D[NR];
    auto done_after = [](int cells_blended) { return __int_as_float((int)0x80000000 | (cells_blended + 1)); };
#pragma unroll
    for (int q = 0; q < PPL; ++q)
        T[q] = xs[q & 1] < V.W && ys[q >> 1] < V.H && !(1.0f < bp.eps) ? 1.0f : done_after(0);
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) N0[rr] = N1[rr] = N2[rr] = D[rr] = make_float2(0.f, 0.f);
    CellBatches feed(cells, rec + V.rec_base * kRecF4, rg.y, K, lane);
    feed.read_ids(rg.x, K, lane);
    feed.issue(s_rec[0], rg.x, K, lane);
    cp_async_commit();
    feed.read_ids(rg.x + CB, K, lane);
    int buf = 0;
    for (uint32_t e = rg.x; e < rg.y; e += CB, buf ^= 1) {
        // before cell n a pixel stops if T_n < eps (Sec. V-B)
        bool all = true;
#pragma unroll
        for (int q = 0; q < PPL; ++q) all = all && T[q] < bp.eps;
        if (__all_sync(0xffffffffu, all)) break;
        feed.issue(s_rec[buf ^ 1], e + CB, K, lane);  // (that buffer's batch was read in the last iteration)
        cp_async_commit();
        feed.read_ids(e + 2 * CB, K, lane);
        cp_async_wait<1>();
        __syncwarp();
        const float4 *r = s_rec[buf];
        const bool mine = lane < K * feed.count(e, K);  // lane l: the batch's l-th Gaussian
        const float4 rl = r[kRecF4 * lane];
        unsigned hits = __ballot_sync(0xffffffffu, mine && touches_rows(rl, bx0, by0, (float)ROWS));
        // Gaussians whose box holds the whole sub-tile: no per-pixel test
        const unsigned full = VAR ? 0u : __ballot_sync(0xffffffffu, mine && covers_rows(rl, bx0, by0, (float)ROWS));
        const float amin = VAR && (bp.flags & DGS_FLAG_ALPHA_SKIP) ? 1.0f / 255.0f : 0.0f;
        // an opacity below the clamp keeps every alpha there (G' <= 1, to the last
        // bits): batches without a larger one in reach go without the minimum
        const bool clamp = VAR || (hits & __ballot_sync(0xffffffffu, !(r[kRecF4 * lane + 1].w < 0.9999f * bp.alpha_max))) != 0u;
        auto blend_batch = [&](auto with_clamp) {
        while (hits) {
            // the next cell with a Gaussian in reach: cell c of the batch, its Gaussians' lanes in mask
            const int c = KT > 0 ? (__ffs(hits) - 1) / K : (int)((unsigned)(__ffs(hits) - 1) * kinv >> 16);
            unsigned mask = hits & (kmask << (c * K));
            hits ^= mask;
            const float v = r[kRecF4 * (c * K) + 2].w;
            float2 A0[NR], A1[NR], A2[NR], B[NR], P[NR];
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                A0[rr] = A1[rr] = A2[rr] = B[rr] = make_float2(0.f, 0.f);
                P[rr] = make_float2(1.0f, 1.0f);
            }
            const float2 nv2 = make_float2(-v, -v);
            for (; mask; mask &= mask - 1) {
                const int k = __ffs(mask) - 1;
                const float4 r0 = r[3 * k], r1 = r[3 * k + 1], r2 = r[3 * k + 2];
                // offsets of the two columns, and of the rows (packed where there are two)
                float dx[2], dy[NR], s22[NR];
                {
                    const float2 d = __fadd2_rn(make_float2(pxs[0], pxs[1]), make_float2(-r0.x, -r0.x));
                    dx[0] = d.x;
                    dx[1] = d.y;
                }
                if (NR == 2) {
                    const float2 d = __fadd2_rn(make_float2(pys[0], pys[NR - 1]), make_float2(-r0.y, -r0.y));
                    dy[0] = d.x;
                    dy[NR - 1] = d.y;
                } else {
                    dy[0] = pys[0] - r0.y;
                }
                bool h[PPL];
                if (VAR || !((full >> k) & 1u)) {  // (else every pixel of the sub-tile is in the box)
                    bool hx[2], hy[NR];
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2) hx[c2] = fabsf(dx[c2]) <= r0.z;
#pragma unroll
                    for (int rr = 0; rr < NR; ++rr) hy[rr] = fabsf(dy[rr]) <= r0.w;
                    if (VAR) {
#pragma unroll
                        for (int q = 0; q < PPL; ++q) h[q] = !(T[q] < bp.eps) && hx[q & 1] && hy[q >> 1];
                    } else {
                        // outside the box along a column or a row: an offset far off
                        // the Gaussian, so exp2 gives alpha = +0 exactly (a done pixel
                        // takes the cell's sums with weight 0: records are finite,
                        // gauss_record)
#pragma unroll
                        for (int c2 = 0; c2 < 2; ++c2) dx[c2] = hx[c2] ? dx[c2] : kFar;
#pragma unroll
                        for (int rr = 0; rr < NR; ++rr) dy[rr] = hy[rr] ? dy[rr] : kFar;
                    }
                }
                const float2 pdx = __fmul2_rn(make_float2(r1.x, r1.x), make_float2(dx[0], dx[1]));
                {
                    const float2 s2 = __fmul2_rn(make_float2(r1.z, r1.z), make_float2(dy[0], dy[NR - 1]));
                    const float2 q = __fmul2_rn(s2, s2);
                    s22[0] = q.x;
                    s22[NR - 1] = NR == 2 ? q.y : q.x;
                }
#pragma unroll
                for (int rr = 0; rr < NR; ++rr) {
                    const float dyq = dy[rr];
                    const float2 s1 = __ffma2_rn(make_float2(r1.y, r1.y), make_float2(dyq, dyq), pdx);
                    const float2 qd = __ffma2_rn(s1, s1, make_float2(s22[rr], s22[rr]));
                    float2 al = __fmul2_rn(make_float2(r1.w, r1.w), make_float2(ex2_approx(-qd.x), ex2_approx(-qd.y)));
                    // a pixel the Gaussian does not reach (or, with the alpha skip, an
                    // alpha below 1/255) takes alpha 0: every update below leaves it unchanged
                    if (VAR) {
                        al.x = h[2 * rr] && al.x >= amin ? fminf(al.x, bp.alpha_max) : 0.f;
                        al.y = h[2 * rr + 1] && al.y >= amin ? fminf(al.y, bp.alpha_max) : 0.f;
                    } else if (decltype(with_clamp)::value) {
                        al.x = fminf(al.x, bp.alpha_max);
                        al.y = fminf(al.y, bp.alpha_max);
                    }
                    A0[rr] = __ffma2_rn(al, make_float2(r2.x, r2.x), A0[rr]);
                    A1[rr] = __ffma2_rn(al, make_float2(r2.y, r2.y), A1[rr]);
                    A2[rr] = __ffma2_rn(al, make_float2(r2.z, r2.z), A2[rr]);
                    B[rr] = __fadd2_rn(B[rr], al);
                    P[rr] = __ffma2_rn(P[rr], __fmul2_rn(nv2, al), P[rr]);
                }
            }
            const float now_done = done_after((int)(e - rg.x) + c + 1);
            const bool exclude = VAR && (bp.flags & DGS_FLAG_TERM_EXCLUDE) != 0;
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                const float2 Tr = make_float2(T[2 * rr], T[2 * rr + 1]);
                float2 w = __fmul2_rn(make_float2(v, v), Tr);
                const float2 Tn = __fmul2_rn(Tr, P[rr]);
                const bool d0 = Tr.x < bp.eps, d1 = Tr.y < bp.eps;      // done before this cell
                const bool n0 = Tn.x < bp.eps, n1 = Tn.y < bp.eps;      // (or with it)
                w.x = d0 || (exclude && n0) ? 0.f : w.x;  // exclude, the 3DGS rule: that cell is not blended
                w.y = d1 || (exclude && n1) ? 0.f : w.y;
                N0[rr] = __ffma2_rn(w, A0[rr], N0[rr]);
                N1[rr] = __ffma2_rn(w, A1[rr], N1[rr]);
                N2[rr] = __ffma2_rn(w, A2[rr], N2[rr]);
                D[rr] = __ffma2_rn(w, B[rr], D[rr]);
                const float end = exclude ? done_after((int)(e - rg.x) + c) : now_done;
                T[2 * rr] = d0 ? Tr.x : n0 ? end : Tn.x;
                T[2 * rr + 1] = d1 ? Tr.y : n1 ? end : Tn.y;
            }
        }
        };
        if (clamp) blend_batch(std::true_type{}); else blend_batch(std::false_type{});
        __syncwarp();  // every lane is done with s_rec[buf] before it is refilled
    }
    cp_async_wait<0>();  // copies of entries past an early stop land before the buffers are reused
    __syncwarp();
    const long long HW = (long long)V.W * V.H;
    float *img = V.out ? V.out : out_rgb + 3 * V.pix_base;
    float *im2 = out_rgb2 ? out_rgb2 + 3 * V.pix_base : nullptr;
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        if (!(xs[q & 1] < V.W && ys[q >> 1] < V.H)) continue;
        const long long pin = (long long)ys[q >> 1] * V.W + xs[q & 1];
        const float m0 = q & 1 ? N0[q >> 1].y : N0[q >> 1].x, m1 = q & 1 ? N1[q >> 1].y : N1[q >> 1].x;
        const float m2 = q & 1 ? N2[q >> 1].y : N2[q >> 1].x, Dq = q & 1 ? D[q >> 1].y : D[q >> 1].x;
        float c0, c1, c2;
        if (VAR && (bp.flags & DGS_FLAG_NUMERATOR)) {  // the numerator of Eq. 12
            c0 = m0; c1 = m1; c2 = m2;
        } else if (VAR) {  // Eq. 12, with a background weight (N + w_bg bg) / (D + w_bg)
            const float Dp = Dq + bp.w_bg;
            const bool hit = Dp > bp.d_min;
            c0 = hit ? (m0 + bp.w_bg * bp.bg0) / Dp : bp.bg0;
            c1 = hit ? (m1 + bp.w_bg * bp.bg1) / Dp : bp.bg1;
            c2 = hit ? (m2 + bp.w_bg * bp.bg2) / Dp : bp.bg2;
        } else {  // Eq. 12
            const bool hit = Dq > bp.d_min;
            c0 = hit ? m0 / Dq : bp.bg0;
            c1 = hit ? m1 / Dq : bp.bg1;
            c2 = hit ? m2 / Dq : bp.bg2;
        }
        img[pin] = c0;
        img[HW + pin] = c1;
        img[2 * HW + pin] = c2;
        if (im2) {
            im2[pin] = c0;
            im2[HW + pin] = c1;
            im2[2 * HW + pin] = c2;
        }
        out_D[V.pix_base + pin] = Dq;
        out_nd[V.pix_base + pin] = T[q] < bp.eps ? (__float_as_int(T[q]) & 0x7fffffff) - 1 : (int)(rg.y - rg.x);
    }
}

template <int KT, int PPL, bool VAR>
__global__ void __launch_bounds__(WT, fwd_minb(VAR)) k_blend_fwd(const ViewDesc *__restrict__ views, int n_views,
                                                  const uint32_t *__restrict__ order,
                                                  const uint2 *__restrict__ ranges, const uint32_t *__restrict__ cells,
                                                  const float4 *__restrict__ rec, BlendParams bp,
                                                  float *__restrict__ out_rgb, float *__restrict__ out_rgb2,
                                                  float *__restrict__ out_D, int *__restrict__ out_nd) {
    __shared__ float4 s_rec[FSTAGE][kBatchF4];
    chain_wait();
    blend_fwd_unit<KT, PPL, VAR>(blockIdx.x, views, n_views, order, ranges, cells, rec, bp, out_rgb, out_rgb2, out_D, out_nd,
                                s_rec);
}

// Persistent form for chains whose sizes live on the device: a fixed grid of
// exactly the resident warps pulls sub-tiles from an atomic counter (*work
// starts at 0) until the chain's total_tiles * FWD_SUB units are taken, so the
// dense and the empty regions of the images balance dynamically.  One
// atomic per sub-tile: their rate is bounded by the blend work between them.
template <int KT, bool VAR>
__global__ void __launch_bounds__(WT, fwd_minb(VAR)) k_blend_fwd_pull(const ViewDesc *__restrict__ views,
                                                       const uint32_t *__restrict__ order,
                                                       const uint2 *__restrict__ ranges,
                                                       const uint32_t *__restrict__ cells,
                                                       const float4 *__restrict__ rec, BlendParams bp,
                                                       float *__restrict__ out_rgb, float *__restrict__ out_D,
                                                       int *__restrict__ out_nd, const ChainSizes *__restrict__ dsz,
                                                       uint32_t *__restrict__ work) {
    __shared__ float4 s_rec[FSTAGE][kBatchF4];
    chain_wait();
    const int n_views = dsz->n_views;
    const uint32_t units = (uint32_t)dsz->total_tiles * FWD_SUB;
    for (;;) {
        uint32_t u = 0;
        if (threadIdx.x == 0) u = atomicAdd(work, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= units) break;
        blend_fwd_unit<KT, FWD_PPL, VAR>((int)u, views, n_views, order, ranges, cells, rec, bp, out_rgb, nullptr, out_D, out_nd,
                                    s_rec);
        __syncwarp();
    }
}

// Do the blend kernels need their variant form (a flag, a background weight, or
// no dilation)?  The default form gives a pixel outside a Gaussian's box an offset of
// kFar, and needs L's entries finite for it: with the screen covariance dilated they
// are at most 1/sqrt(dilation), without, a Gaussian of no extent has infinite ones.
// The variant form masks every pixel's alpha instead.
static bool blend_variants(const BlendParams &bp) {
    return (bp.flags & (DGS_FLAG_ALPHA_SKIP | DGS_FLAG_TERM_EXCLUDE | DGS_FLAG_NUMERATOR)) != 0 || bp.w_bg != 0.f ||
           bp.dilation < 1e-12f;
}

template <int KT, bool VAR>
static unsigned pull_grid(int total_tiles) {
    const long long per_grid = resident_ctas((const void *)k_blend_fwd_pull<KT, VAR>, WT);
    return (unsigned)std::min<long long>((long long)total_tiles * FWD_SUB, per_grid);
}

void launch_blend_fwd(const ViewDesc *views, int n_views, int total_tiles, const uint32_t *order, const uint2 *ranges,
                      const uint32_t *tile_cells, const float4 *rec, const BlendParams &bp, float *out_rgb,
                      float *out_rgb2, float *out_D, int *out_nd, int K_all, cudaStream_t st,
                      const ChainSizes *dsz, uint32_t *work) {
    if (total_tiles == 0) return;
    if (dsz) {
        // exactly the resident warps
#define DGS_PULL(KV, VV)                                                                                     \
        launch_chained(k_blend_fwd_pull<KV, VV>, pull_grid<KV, VV>(total_tiles), WT, 0, st, views, order, ranges, tile_cells, \
                       rec, bp, out_rgb, out_D, out_nd, dsz, work)
        if (blend_variants(bp)) {
            switch (K_all) {
                case 8: DGS_PULL(8, true); break;
                case 10: DGS_PULL(10, true); break;
                default: DGS_PULL(0, true); break;
            }
        } else {
            switch (K_all) {
                case 8: DGS_PULL(8, false); break;
                case 10: DGS_PULL(10, false); break;
                default: DGS_PULL(0, false); break;
            }
        }
#undef DGS_PULL
        return;
    }
#define DGS_FWD(KV, PV, VV)                                                                                  \
    launch_chained(k_blend_fwd<KV, PV, VV>, (unsigned)total_tiles * (kTile / (2 * PV)), WT, 0, st, views, n_views, order, \
                   ranges, tile_cells, rec, bp, out_rgb, out_rgb2, out_D, out_nd)
    if (blend_variants(bp)) {
        switch (K_all) {
            case 8: DGS_FWD(8, FWD_PPL, true); break;
            case 10: DGS_FWD(10, FWD_PPL, true); break;
            default: DGS_FWD(0, FWD_PPL, true); break;
        }
    } else if (total_tiles <= kFewTiles) {
        switch (K_all) {
            case 8: DGS_FWD(8, 2, false); break;
            case 10: DGS_FWD(10, 2, false); break;
            default: DGS_FWD(0, 2, false); break;
        }
    } else {
        switch (K_all) {
            case 8: DGS_FWD(8, FWD_PPL, false); break;
            case 10: DGS_FWD(10, FWD_PPL, false); break;
            default: DGS_FWD(0, FWD_PPL, false); break;
        }
    }
#undef DGS_FWD
}

// ---------------------------------------------------------------- counters
// Diagnostic replay of the AABB tests (no blending): per pixel, the
// (pixel, Gaussian) pairs of blended cells, those passing the AABB test, and
// the passing pairs over the whole tile list.  counts[0..3] as in dgs_counts.
__global__ void __launch_bounds__(BT) k_count_pairs(const ViewDesc *__restrict__ views, int n_views,
                                                    const uint2 *__restrict__ ranges, const uint32_t *__restrict__ cells,
                                                    const float4 *__restrict__ rec, const int *__restrict__ ndpix,
                                                    unsigned long long *__restrict__ counts) {
    __shared__ int s_view;
    const int tid = threadIdx.x, tile = blockIdx.x;
    if (tid == 0) s_view = find_view(views, n_views, tile);
    __syncthreads();
    const ViewDesc &V = views[s_view];
    const int local = tile - V.tile_base;
    const int tx = local % V.Tx, ty = local / V.Tx;
    const int xi = tx * kTile + (tid & (kTile - 1)), yi = ty * kTile + (tid >> 4);
    unsigned long long c[4] = {0, 0, 0, 0};
    if (xi < V.W && yi < V.H) {
        const int nd = ndpix[V.pix_base + (long long)yi * V.W + xi];
        const float px = (float)xi + 0.5f, py = (float)yi + 0.5f;
        const uint2 rg = ranges[tile];
        const float4 *vrec = rec + V.rec_base * kRecF4;
        for (uint32_t e = rg.x; e < rg.y; ++e) {
            const bool blended = (int)(e - rg.x) < nd;
            const float4 *r = vrec + (long long)cells[e] * V.K * kRecF4;
            unsigned in = 0;
            for (int k = 0; k < V.K; ++k) {
                const float4 r0 = __ldg(r + 3 * k);
                in += (fabsf(px - r0.x) <= r0.z && fabsf(py - r0.y) <= r0.w) ? 1u : 0u;
            }
            c[2] += in;
            if (blended) { c[0] += V.K; c[1] += in; c[3] += 1; }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        unsigned long long v = c[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0 && v) atomicAdd(counts + i, v);
    }
}

void launch_count_pairs(const ViewDesc *views, int n_views, int total_tiles, const uint2 *ranges,
                        const uint32_t *tile_cells, const float4 *rec, const int *nd, unsigned long long *counts,
                        cudaStream_t st) {
    if (total_tiles == 0) return;
    k_count_pairs<<<total_tiles, BT, 0, st>>>(views, n_views, ranges, tile_cells, rec, nd, counts);
}

// ---------------------------------------------------------------- adjoint
// With C = N/D and g = dL/dC:  dN = g/D, dD = -(g.C)/D.  Writing
// x_n = v_n T_n (dN.A_n + dD B_n), C's degree-0 homogeneity in the weights
// gives sum_n x_n = 0 over the blended cells, so the total gradient through
// the transmittance of all LATER cells, S_n = sum_{m>n} x_m, equals
// -sum_{m<=n} x_m and is known front to back: the replay needs no division
// by T and stores no per-cell state.  Per Gaussian k of cell n at a pixel:
//     dL/dalpha = v T_n (dN.c_k + dD) - v S_n / (1 - v alpha)
//     dL/dc_k   = v T_n alpha dN
//     dL/dv_n   = T_n (dN.A_n + dD B_n) - S_n sum_k alpha_k / (1 - v alpha_k)
// then alpha = sigma G' (unless clamped) and G' = exp(-q/2).
//
// Same work unit as the forward (one warp per sub-tile).  Per cell, the warp
// replays its pixels keeping G' of the Gaussians that reach the sub-tile in
// warp-private shared memory and updates S and T; then groups of eight lanes take
// a Gaussian each and sum its nine screen-space gradient terms over the
// sub-tile's pixels, and the totals are added to global memory (one
// atomic add per value per sub-tile): see k_blend_bwd.

// Sums of eight per-lane values over the eight lanes of a group (lanes that
// differ in bits 0..2): three halving steps (offsets 4, 2, 1) in which each
// lane keeps half of its values and receives its partner's other half, so
// lane L ends with the group's total of value group_owner8(L): 7 shuffles
// instead of 8 x 3.
__device__ __forceinline__ float group_sum8(float v[8], int lane) {
#pragma unroll
    for (int step = 0; step < 3; ++step) {
        const int bit = 4 >> step;
        const bool hi = lane & bit;
#pragma unroll
        for (int i = 0; i < (4 >> step); ++i) {
            const float keep = hi ? v[2 * i + 1] : v[2 * i];
            const float send = hi ? v[2 * i] : v[2 * i + 1];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
    }
    return v[0];
}

__device__ __forceinline__ int group_owner8(int lane) {
    return ((lane >> 2) & 1) + ((lane >> 1) & 1) * 2 + (lane & 1) * 4;
}

__device__ __forceinline__ float warp_sum(float a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// 1/x to ~1 ulp (MUFU); x = 1 - v alpha >= 1 - alpha_max here
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One lane's sums of a Gaussian's screen-space gradient terms over its pixels
// (components x, y: its two columns; e the pixel's dL/dN):
//   dop = sum dG                 (dsigma)
//   Y, Q = sum dG dy, sum dG dy^2  (times sigma: the moments of dq' = -2 dL/dq;
//          the dx-weighted ones follow per column at the end)
//   C    = sum v T alpha e, less the factor `colour` (drgb)
//   dv   = sum -S_n alpha / (1 - v alpha), less the same factor (dL/dv_n's share)
struct LaneGrad {
    float2 dop, Y, Q, C0, C1, C2, dv;
};

// A Gaussian's terms at one pixel pair of a row: G' = Gv, F = v T_n (e0, e1,
// e2, eD), nS = -v S_n (WV: -S_n) of the pixels.  With dalpha = v T_n (e.c +
// eD) - v S_n / (1 - v alpha):  dG = dalpha G', zero where alpha is clamped.
// CLAMP = false: sigma < alpha_max, so alpha = sigma G' nowhere reaches the
// clamp; sigma is then applied to the sums instead of to each pixel.
template <bool CLAMP, bool WV>
__device__ __forceinline__ void pair_grad2(LaneGrad &a, float2 Gv, float2 F0, float2 F1, float2 F2, float2 FD, float2 nS,
                                           float dy, float op, float v, float nvop, float4 r2, float alpha_max) {
    float2 al = Gv, om, raw;
    if (CLAMP) {
        raw = __fmul2_rn(make_float2(op, op), Gv);
        al = make_float2(fminf(raw.x, alpha_max), fminf(raw.y, alpha_max));
        om = __ffma2_rn(make_float2(-v, -v), al, make_float2(1.0f, 1.0f));
    } else {
        om = __ffma2_rn(make_float2(nvop, nvop), Gv, make_float2(1.0f, 1.0f));
    }
    const float2 rom = make_float2(rcp_approx(om.x), rcp_approx(om.y));
    const float2 u = __ffma2_rn(F0, make_float2(r2.x, r2.x),
                                __ffma2_rn(F1, make_float2(r2.y, r2.y), __ffma2_rn(F2, make_float2(r2.z, r2.z), FD)));
    float2 dal;
    if (WV) {
        const float2 w = __fmul2_rn(nS, rom);
        a.dv = __ffma2_rn(w, al, a.dv);
        dal = __ffma2_rn(make_float2(v, v), w, u);
    } else {
        dal = __ffma2_rn(nS, rom, u);
    }
    a.C0 = __ffma2_rn(F0, al, a.C0);
    a.C1 = __ffma2_rn(F1, al, a.C1);
    a.C2 = __ffma2_rn(F2, al, a.C2);
    float2 dG = __fmul2_rn(dal, Gv);
    if (CLAMP) {
        dG.x = raw.x < alpha_max ? dG.x : 0.f;
        dG.y = raw.y < alpha_max ? dG.y : 0.f;
    }
    const float dy2 = dy * dy;
    a.dop = __fadd2_rn(a.dop, dG);
    a.Y = __ffma2_rn(dG, make_float2(dy, dy), a.Y);
    a.Q = __ffma2_rn(dG, make_float2(dy2, dy2), a.Q);
}

// The mean's terms of a lane, from its moments m = sum dq' (dx, dy): with the
// record's L scaled by kappa (kappa^2 = log2(e)/2), q = |L^T d|^2 and
// dq/dmu = -2 Q d = -(2/kappa^2) L (s1, s2), (s1, s2) = L^T d = (p dx + r dy,
// t dy), 2/kappa^2 = 4 ln 2; summed over pixels, sum dq' L (s1, s2) =
// (p u, r u + t^2 m_y) with u = p m_x + r m_y (linear in the moments, so each
// lane converts its partial sums before the warp reduction: no shuffle).
__device__ __forceinline__ void mean_terms(float4 r1, float &a0, float &a1) {
    const float u = fmaf(r1.x, a0, r1.y * a1);
    const float b1 = fmaf(r1.y, u, r1.z * r1.z * a1);
    a0 = r1.x * u;
    a1 = b1;
}

// Constant factor of reduction slot j: dL/dq = -dq'/2, so
// dmu = -(4 ln 2)(-1/2) acc = 2 ln 2 acc, da = -acc/2, db = -acc (the 2 dx dy
// term), dc = -acc/2; rgb unchanged.
__device__ __forceinline__ float slot_scale(int j) {
    return j < 2 ? 2.0f * LN2 : (j == 3 ? -1.0f : (j < 5 ? -0.5f : 1.0f));
}

// screen-space gradient slot (of kGradF) that reduction slot j feeds
__device__ __forceinline__ int grad_slot(int j) { return j < 5 ? j : j + 1; }

// The adjoint's work unit: one warp per 16 x (2 PPL) sub-tile, pixels of a
// lane as in the forward (lane_col, lane_row).  Per cell:
//   pass 1, pixel-major (a lane owns four pixels): replays the forward, keeping
//     G' of the Gaussians that reach the sub-tile in warp-private shared memory
//     (one row of 128 pixels each), and updates T and S; then the lanes leave
//     their pixels' factors v T_n e and -v S_n there too;
//   pass 2, Gaussian-major: four Gaussians at a time, eight lanes each; a lane
//     takes columns w and w + 8 of all eight rows (16 pixels) of its Gaussian
//     and sums its terms in registers, so one reduction over eight lanes (7 + 3
//     shuffles) serves four Gaussians and 32 totals leave in one atomic add per
//     lane.  Of the last one or two Gaussians of a cell each gets 32 or 16 lanes.
// Bound by instruction issue and the shared-memory data path together (189
// warp instructions and 58 wavefronts per (sub-tile, Gaussian), 66% and 75% of
// their peaks before the split of the last round).  A pixel-major pass 2 needs
// a 32-lane reduction of nine values per Gaussian (229 instructions): 6.33 ms
// on the 1M-Gaussian 8-view step against 5.17 ms; always four groups: 5.72 ms
// there, and 1.50 against 1.27 ms where cells have few hits (neural cells, 1.6
// per cell and sub-tile); two Gaussians per lane (half the factor loads): 5.62 ms,
// its registers leave 16 warps an SM.
constexpr int BWD_PPL = 4;
// Resident one-warp CTAs per SM the register budget is set for: 22 are what the
// shared memory of K = 10 admits (80 registers; 20 at 96 registers is 4% slower
// on the 1M-Gaussian step).  With dL/dv_n's sums 80 registers spill: 20 there
// (0.43 against 0.47 ms on 20,011 cells x 5, three 641 x 479 views).
constexpr int bwd_minb(bool wv) { return wv ? 20 : 22; }

// float4s of shared memory: records [NSTAGE][3 K], G' rows [K][32] (a lane's PPL
// pixels), v T_n (e0, e1) and v T_n (e2, eD) [PPL / 2][32] each, -v S_n
// [32] (PPL), and the Gaussian of every row (K ints)
__host__ __device__ constexpr int bwd_smem_f4(int K, int PPL) {
    return NSTAGE * kRecF4 * K + WT * K * PPL / 4 + WT * PPL + WT * PPL / 4 + (K + 3) / 4;
}

// A lane's pixels in shared memory, one pair per lane row: 16 or 8 bytes.
template <int NR> struct RowPairs;
template <> struct RowPairs<2> {
    using T = float4;
    static __device__ __forceinline__ T pack(const float2 (&v)[2]) { return make_float4(v[0].x, v[0].y, v[1].x, v[1].y); }
    static __device__ __forceinline__ float2 row(T t, int rr) { return rr == 0 ? make_float2(t.x, t.y) : make_float2(t.z, t.w); }
};
template <> struct RowPairs<1> {
    using T = float2;
    static __device__ __forceinline__ T pack(const float2 (&v)[1]) { return v[0]; }
    static __device__ __forceinline__ float2 row(T t, int) { return t; }
};

template <int KT, int PPL, bool VAR, bool WV>
__global__ void __launch_bounds__(WT, bwd_minb(WV)) k_blend_bwd(const ViewDesc *__restrict__ views, int n_views,
                                                  const uint32_t *__restrict__ order,
                                                  const uint2 *__restrict__ ranges, const uint32_t *__restrict__ cells,
                                                  const float4 *__restrict__ rec, BlendParams bp,
                                                  const float *__restrict__ rgb, const float *__restrict__ Dpix,
                                                  const int *__restrict__ ndpix, const float *__restrict__ dL_drgb,
                                                  float *__restrict__ g2d, float *__restrict__ g_cell_v) {
    extern __shared__ float4 s_bwd[];
    chain_wait();
    const int lane = threadIdx.x;
    constexpr int NR = PPL / 2, ROWS = 2 * PPL, NSUB = kTile / ROWS;  // rows per lane (pixel mapping as in the forward)
    using Pairs = RowPairs<NR>;
    const int tile = (int)order[blockIdx.x / NSUB], sub = blockIdx.x % NSUB;
    const int vi = find_view(views, n_views, tile);
    const ViewDesc &V = views[vi];
    const int K = KT > 0 ? KT : V.K;
    const int per = kRecF4 * K;
    float4 *const s_rec = s_bwd;                    // [NSTAGE][per]
    typename Pairs::T *const s_G = reinterpret_cast<typename Pairs::T *>(s_rec + NSTAGE * per);  // [K][WT]
    float4 *const s_F01 = reinterpret_cast<float4 *>(s_G + WT * K);  // [NR][WT]
    float4 *const s_F2D = s_F01 + NR * WT;                           // [NR][WT]
    typename Pairs::T *const s_nS = reinterpret_cast<typename Pairs::T *>(s_F2D + NR * WT);  // [WT]
    int *const s_k = reinterpret_cast<int *>(s_nS + WT);  // [K]
    const int local = tile - V.tile_base;
    const int tx = local % V.Tx, ty = local / V.Tx;
    const float bx0 = (float)(tx * kTile), by0 = (float)(ty * kTile + ROWS * sub);
    int xs[2], ys[NR];
    float pxs[2], pys[NR];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        xs[c] = tx * kTile + lane_col(lane, c);
        pxs[c] = (float)xs[c] + 0.5f;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        ys[r] = ty * kTile + ROWS * sub + lane_row(lane, r);
        pys[r] = (float)ys[r] + 0.5f;
    }
    const long long HW = (long long)V.W * V.H;

    // Per pixel: dL/dN = e, dL/dD = eD, and S's start value, the sum of x_n
    // over the processed cells: 0 for C = N / D (degree-0 homogeneity), else
    // w_bg g.(C - bg) / (D + w_bg) with a background weight, g.C for the
    // numerator output (dL/dN = g, dL/dD = 0).
    int nd[PPL];
    float e0s[PPL], e1s[PPL], e2s[PPL], eDs[PPL], S0[PPL];
    int ndm = 0;
    const bool numer = VAR && (bp.flags & DGS_FLAG_NUMERATOR) != 0;
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        nd[q] = 0;
        e0s[q] = e1s[q] = e2s[q] = eDs[q] = S0[q] = 0.f;
        if (xs[q & 1] < V.W && ys[q >> 1] < V.H) {
            const long long pin = (long long)ys[q >> 1] * V.W + xs[q & 1];
            const float Dp = VAR ? Dpix[V.pix_base + pin] + bp.w_bg : Dpix[V.pix_base + pin];
            if (numer || Dp > bp.d_min) {
                nd[q] = ndpix[V.pix_base + pin];
                const float *gi = dL_drgb + 3 * V.pix_base;
                const float *ci = rgb + 3 * V.pix_base;
                const float g0 = gi[pin], g1 = gi[HW + pin], g2 = gi[2 * HW + pin];
                const float c0 = ci[pin], c1 = ci[HW + pin], c2 = ci[2 * HW + pin];
                if (numer) {
                    e0s[q] = g0; e1s[q] = g1; e2s[q] = g2;
                    S0[q] = g0 * c0 + g1 * c1 + g2 * c2;
                } else {
                    const float iD = 1.0f / Dp;
                    e0s[q] = g0 * iD; e1s[q] = g1 * iD; e2s[q] = g2 * iD;
                    eDs[q] = -(g0 * c0 + g1 * c1 + g2 * c2) * iD;
                    if (VAR) S0[q] = bp.w_bg * (g0 * (c0 - bp.bg0) + g1 * (c1 - bp.bg1) + g2 * (c2 - bp.bg2)) * iD;
                }
            }
        }
        ndm = max(ndm, nd[q]);
    }
    // the lane's pixels as row pairs (columns 0 and 1 of lane row rr)
    float2 e0[NR], e1[NR], e2[NR], eD[NR], T[NR], S[NR];
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) {
        e0[rr] = make_float2(e0s[2 * rr], e0s[2 * rr + 1]);
        e1[rr] = make_float2(e1s[2 * rr], e1s[2 * rr + 1]);
        e2[rr] = make_float2(e2s[2 * rr], e2s[2 * rr + 1]);
        eD[rr] = make_float2(eDs[2 * rr], eDs[2 * rr + 1]);
        T[rr] = make_float2(nd[2 * rr] > 0 ? 1.0f : 0.f, nd[2 * rr + 1] > 0 ? 1.0f : 0.f);
        S[rr] = make_float2(S0[2 * rr], S0[2 * rr + 1]);
    }
    const int ndmax = __reduce_max_sync(0xffffffffu, ndm);
    const uint2 rg = ranges[tile];
    const uint32_t end = rg.x + min((uint32_t)ndmax, rg.y - rg.x);
    const float4 *vrec = rec + V.rec_base * kRecF4;

    // pass 2's lane: group (Gaussian of four) and columns; the reduction slot it ends up with
    const int grp = lane >> 3, w8 = lane & 7;
    const float2 px2 = make_float2(bx0 + (float)w8 + 0.5f, bx0 + (float)w8 + 8.5f);
    const int slot = group_owner8(lane);

    CellFeed feed{cells, rg.x, end, 0u};
#pragma unroll
    for (int b = 0; b < NSTAGE - 1; ++b) {
        if (rg.x + b < end) issue_cell<KT>(s_rec + b * per, vrec, feed.id(rg.x + b, lane), per, lane);
        cp_async_commit();
    }
    int buf = 0;
    for (uint32_t e = rg.x; e < end; ++e) {
        const int fill = buf == 0 ? NSTAGE - 1 : buf - 1;  // the buffer of entry e - 1, read by now
        if (e + NSTAGE - 1 < end) issue_cell<KT>(s_rec + fill * per, vrec, feed.id(e + NSTAGE - 1, lane), per, lane);
        cp_async_commit();
        cp_async_wait<NSTAGE - 1>();
        __syncwarp();
        const int n = (int)(e - rg.x);
        const float4 *r = s_rec + buf * per;
        buf = buf == NSTAGE - 1 ? 0 : buf + 1;
        const float v = r[2].w;
        // the Gaussians that reach the sub-tile: row i of G' belongs to the i-th
        const unsigned hits = __ballot_sync(0xffffffffu, lane < K && touches_rows(r[kRecF4 * lane], bx0, by0, (float)ROWS));
        const int rows = __popc(hits);
        if ((hits >> lane) & 1u) s_k[__popc(hits & ((1u << lane) - 1u))] = lane;
        // With v <= 1 every 1 - v alpha is at least 1 - alpha_max, and the zero
        // factors of a finished pixel (T = S = 0) alone keep it out of pass 2;
        // otherwise the reciprocal may be infinite and its G' is zeroed too.
        const bool mask_G = !VAR && !(v <= 1.0f);
        if (rows == 0) {  // (uniform) X = 0, P = 1: only a finished pixel changes
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                T[rr].x = n + 1 < nd[2 * rr] ? T[rr].x : 0.f;
                T[rr].y = n + 1 < nd[2 * rr + 1] ? T[rr].y : 0.f;
            }
            __syncwarp();  // every lane is done with the records before they are refilled
            continue;
        }
        // pass 1: replay the cell, keep G'; per pixel P_n and
        // X_n = dN.A_n + dD B_n = sum_k alpha_k (dN.c_k + dD)
        float2 X[NR], P[NR];
        const float2 v2 = make_float2(v, v);
        const float amin = VAR && (bp.flags & DGS_FLAG_ALPHA_SKIP) ? 1.0f / 255.0f : 0.0f;
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) { X[rr] = make_float2(0.f, 0.f); P[rr] = make_float2(1.0f, 1.0f); }
        typename Pairs::T *row = s_G + lane;
#pragma unroll 1
        for (unsigned mask = hits; mask; mask &= mask - 1, row += WT) {
            const int k = __ffs(mask) - 1;
            const float4 r0 = r[3 * k], r1 = r[3 * k + 1], r2 = r[3 * k + 2];
            float dx[2], dy[NR];
            bool hx[2], hy[NR];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                dx[c] = pxs[c] - r0.x;
                hx[c] = fabsf(dx[c]) <= r0.z;
                // outside the box along a column or a row: an offset far off the
                // Gaussian (G' = +0 exactly, as in the forward)
                if (!VAR) dx[c] = hx[c] ? dx[c] : kFar;
            }
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                dy[rr] = pys[rr] - r0.y;
                hy[rr] = fabsf(dy[rr]) <= r0.w;
                if (!VAR) dy[rr] = hy[rr] ? dy[rr] : kFar;
            }
            const float2 pdx = __fmul2_rn(make_float2(r1.x, r1.x), make_float2(dx[0], dx[1]));
            float2 gq[NR];
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                const float dyq = dy[rr];
                const float s2 = r1.z * dyq, s22 = s2 * s2;
                const float2 s1 = __ffma2_rn(make_float2(r1.y, r1.y), make_float2(dyq, dyq), pdx);
                const float2 qd = __ffma2_rn(s1, s1, make_float2(s22, s22));
                float2 Gv = make_float2(ex2_approx(-qd.x), ex2_approx(-qd.y));
                float2 rw = __fmul2_rn(make_float2(r1.w, r1.w), Gv);
                if (VAR) {  // not reached (or alpha skipped, or not a number, as in the forward): G' = 0 leaves X and P as they are
                    if (!(n < nd[2 * rr] && hx[0] && hy[rr] && rw.x >= amin)) Gv.x = rw.x = 0.f;
                    if (!(n < nd[2 * rr + 1] && hx[1] && hy[rr] && rw.y >= amin)) Gv.y = rw.y = 0.f;
                }
                gq[rr] = Gv;
                const float2 al = make_float2(fminf(rw.x, bp.alpha_max), fminf(rw.y, bp.alpha_max));
                const float2 inner = __ffma2_rn(
                    e0[rr], make_float2(r2.x, r2.x),
                    __ffma2_rn(e1[rr], make_float2(r2.y, r2.y), __ffma2_rn(e2[rr], make_float2(r2.z, r2.z), eD[rr])));
                X[rr] = __ffma2_rn(al, inner, X[rr]);
                P[rr] = __ffma2_rn(make_float2(-P[rr].x, -P[rr].y), __fmul2_rn(v2, al), P[rr]);
            }
            if (mask_G) {
#pragma unroll
                for (int rr = 0; rr < NR; ++rr) {
                    gq[rr].x = n < nd[2 * rr] ? gq[rr].x : 0.f;
                    gq[rr].y = n < nd[2 * rr + 1] ? gq[rr].y : 0.f;
                }
            }
            *row = Pairs::pack(gq);
        }
        // per-pixel transmittance bookkeeping (S_n includes x_n; a pixel past its
        // last cell has T = S = 0), and the factors of pass 2.  The cell term of
        // dL/dv, sum over pixels of T_n X_n, joins the Gaussians' terms below so
        // one reduction per cell carries dL/dv.
        float2 dv2 = make_float2(0.f, 0.f), nS[NR];
#pragma unroll
        for (int rr = 0; rr < NR; ++rr) {
            const float2 cA = __fmul2_rn(v2, T[rr]);
            const float2 F0 = __fmul2_rn(cA, e0[rr]), F1 = __fmul2_rn(cA, e1[rr]);
            const float2 F2 = __fmul2_rn(cA, e2[rr]), FD = __fmul2_rn(cA, eD[rr]);
            s_F01[rr * WT + lane] = make_float4(F0.x, F0.y, F1.x, F1.y);
            s_F2D[rr * WT + lane] = make_float4(F2.x, F2.y, FD.x, FD.y);
            if (WV) {
                const float2 TX = __fmul2_rn(T[rr], X[rr]);
                dv2.x += n < nd[2 * rr] ? TX.x : 0.f;
                dv2.y += n < nd[2 * rr + 1] ? TX.y : 0.f;
            }
            const float2 Sn = __ffma2_rn(make_float2(-cA.x, -cA.y), X[rr], S[rr]), Tn = __fmul2_rn(T[rr], P[rr]);
            S[rr].x = n < nd[2 * rr] ? Sn.x : 0.f;
            S[rr].y = n < nd[2 * rr + 1] ? Sn.y : 0.f;
            T[rr].x = n + 1 < nd[2 * rr] ? Tn.x : 0.f;
            T[rr].y = n + 1 < nd[2 * rr + 1] ? Tn.y : 0.f;
            nS[rr] = WV ? make_float2(-S[rr].x, -S[rr].y) : __fmul2_rn(make_float2(-v, -v), S[rr]);
        }
        float dv = dv2.x + dv2.y;
        s_nS[lane] = Pairs::pack(nS);
        __syncwarp();
        const uint32_t cellid = __ldg(cells + e);
        float *gbase = g2d + (V.rec_base + (long long)cellid * K) * kGradF;
        // pass 2: the gradient terms of the rows [c, c + 4 / SPLIT); SPLIT groups of
        // eight lanes share a Gaussian, each taking 8 / SPLIT of the sub-tile's rows
        auto round = [&](auto split, int c) {
            constexpr int SPLIT = decltype(split)::value;
            const int g = grp / SPLIT, part = grp % SPLIT;
            // (three rows left: the fourth group repeats the round's first and drops its sums)
            const bool live = SPLIT > 1 || c + g < rows;
            const int i = live ? c + g : c;
            const int k = s_k[i];
            const typename Pairs::T *Gr = s_G + i * WT + w8;
            const float4 r0 = r[3 * k], r1 = r[3 * k + 1], r2 = r[3 * k + 2];
            const float op = r1.w;
            const float py0 = by0 + 0.5f + (float)part;
            LaneGrad a;
            a.dop = a.Y = a.Q = a.C0 = a.C1 = a.C2 = a.dv = make_float2(0.f, 0.f);
            auto sweep = [&](auto clamp) {
#pragma unroll
                for (int t = 0; t < 4 / SPLIT; ++t) {  // rows j and (with two rows per lane) j + 4
                    const int at = 8 * (SPLIT * t + part) + w8;
                    const typename Pairs::T gp = Gr[at - w8], np = s_nS[at];
#pragma unroll
                    for (int rr = 0; rr < NR; ++rr) {
                        const float4 fa = s_F01[rr * WT + at], fb = s_F2D[rr * WT + at];
                        pair_grad2<decltype(clamp)::value, WV>(
                            a, Pairs::row(gp, rr), make_float2(fa.x, fa.y),
                            make_float2(fa.z, fa.w), make_float2(fb.x, fb.y), make_float2(fb.z, fb.w),
                            Pairs::row(np, rr),
                            (py0 + (float)(SPLIT * t + 4 * rr)) - r0.y, op, v, -v * op, r2, bp.alpha_max);
                    }
                }
            };
            // (not op < alpha_max: a NaN opacity takes the clamp, as in the forward)
            const bool clamp = __any_sync(0xffffffffu, !(op < bp.alpha_max));
            if (clamp) sweep(std::true_type{}); else sweep(std::false_type{});
            const float cs = clamp ? 1.0f : op;
            const float2 dx = __fadd2_rn(px2, make_float2(-r0.x, -r0.x));
            // the lane's totals of slots 0..4 from its per-column sums: with D =
            // sigma dop = sum dq' and Y = sigma Y per column, sum dq' dx = D.dx,
            // sum dq' dx^2 = D.dx^2, sum dq' dx dy = Y.dx
            float acc[8];
            const float2 D = __fmul2_rn(a.dop, make_float2(op, op)), t = __fmul2_rn(D, dx);
            const float2 Y = __fmul2_rn(a.Y, make_float2(op, op));
            acc[0] = t.x + t.y;
            acc[1] = Y.x + Y.y;
            acc[2] = fmaf(t.x, dx.x, t.y * dx.y);
            acc[3] = fmaf(Y.x, dx.x, Y.y * dx.y);
            acc[4] = (a.Q.x + a.Q.y) * op;
            acc[5] = (a.C0.x + a.C0.y) * cs;
            acc[6] = (a.C1.x + a.C1.y) * cs;
            acc[7] = (a.C2.x + a.C2.y) * cs;
            mean_terms(r1, acc[0], acc[1]);
            if (WV) dv += live ? (a.dv.x + a.dv.y) * cs : 0.f;
            float tot = group_sum8(acc, lane), dop = a.dop.x + a.dop.y;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) dop += __shfl_xor_sync(0xffffffffu, dop, o);
#pragma unroll
            for (int o = 8; o < 8 * SPLIT; o <<= 1) {
                tot += __shfl_xor_sync(0xffffffffu, tot, o);
                dop += __shfl_xor_sync(0xffffffffu, dop, o);
            }
            float *gk = gbase + k * kGradF;
            if (live && part == 0) {
                if (tot != 0.f) atomicAdd(gk + grad_slot(slot), tot * slot_scale(slot));
                if (w8 == 0 && dop != 0.f) atomicAdd(gk + 5, dop);
            }
        };
        int c = 0;
#pragma unroll 1
        for (; rows - c > 2; c += 4) round(std::integral_constant<int, 1>{}, c);
        if (rows - c == 2) round(std::integral_constant<int, 2>{}, c);
        if (rows - c == 1) round(std::integral_constant<int, 4>{}, c);
        if (WV) {  // per (view, cell) entry: v_n may differ between views
            dv = warp_sum(dv);
            if (lane == 0 && dv != 0.f) atomicAdd(g_cell_v + V.cell_base + cellid, dv);
        }
        __syncwarp();  // every lane is done with the records and rows before they are refilled
    }
    cp_async_wait<0>();
}

// K_all: K of the chain's scene (compile-time loop for common values; sizes the shared memory)
void launch_blend_bwd(const ViewDesc *views, int n_views, int total_tiles, const uint32_t *order, int K_all, const uint2 *ranges,
                      const uint32_t *tile_cells, const float4 *rec, const BlendParams &bp, const float *rgb,
                      const float *D, const int *nd, const float *dL_drgb, float *g2d, float *g_cell_v,
                      cudaStream_t st) {
    if (total_tiles == 0) return;
#define DGS_BWD(KV, PV, VV)                                                                                      \
    do {                                                                                                        \
        const unsigned grid = (unsigned)total_tiles * (kTile / (2 * PV));                                       \
        const size_t smem = sizeof(float4) * bwd_smem_f4(K_all, PV);                                            \
        if (g_cell_v)                                                                                           \
            launch_chained(k_blend_bwd<KV, PV, VV, true>, grid, WT, smem, st, views, n_views, order, ranges, tile_cells, \
                           rec, bp, rgb, D, nd, dL_drgb, g2d, g_cell_v);                                        \
        else                                                                                                    \
            launch_chained(k_blend_bwd<KV, PV, VV, false>, grid, WT, smem, st, views, n_views, order, ranges, tile_cells, \
                           rec, bp, rgb, D, nd, dL_drgb, g2d, nullptr);                                         \
    } while (0)
    if (blend_variants(bp)) {
        switch (K_all) {
            case 8: DGS_BWD(8, BWD_PPL, true); break;
            case 10: DGS_BWD(10, BWD_PPL, true); break;
            default: DGS_BWD(0, BWD_PPL, true); break;
        }
    } else if (total_tiles <= kFewTiles) {
        switch (K_all) {
            case 8: DGS_BWD(8, 2, false); break;
            case 10: DGS_BWD(10, 2, false); break;
            default: DGS_BWD(0, 2, false); break;
        }
    } else {
        switch (K_all) {
            case 8: DGS_BWD(8, BWD_PPL, false); break;
            case 10: DGS_BWD(10, BWD_PPL, false); break;
            default: DGS_BWD(0, BWD_PPL, false); break;
        }
    }
#undef DGS_BWD
}

}  // namespace dgs
