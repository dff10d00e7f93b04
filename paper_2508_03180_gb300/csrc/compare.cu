// Comparator renderers (the two models Duplex-GS is measured against, Sec.
// III-A; the paper's Tab. VI compares sort lengths): per-Gaussian
// alpha-blending over a global depth order (Eq. 2-3, vanilla 3DGS) and
// sort-free weighted-sum rendering (Eq. 4) with the LC-WSR weight (Eq. 5-6).
// They share the Duplex path's per-Gaussian record, AABB skip, colour, binning
// and radix sort; only the unit that is sorted (every Gaussian instead of
// every cell) and the blending differ.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "blend.cuh"
#include "runtime.h"

namespace dgs {

constexpr int CT = 32;      // threads per work unit (one warp per 16x8 sub-tile)
constexpr int CROWS = 8;
constexpr int CSUB = kTile / CROWS;  // sub-tiles per tile

// One warp per 16x8-pixel sub-tile, four pixels per lane in packed row pairs
// (the hybrid's mapping: lane_col, lane_row).  The tile's Gaussians are taken 32 at
// a time: their records arrive in shared memory by asynchronous copies one
// batch ahead, a ballot keeps those whose AABB reaches the sub-tile (a second one
// those that hold all of it and need no test per pixel), and the warp walks them in
// list order (depth order for alpha-blending).
//   ALPHA: C += T alpha c, T *= 1 - alpha; a pixel stops before the entry at
//          which T < eps (the cell rule of the hybrid renderer at K = 1);
//          out = C + T bg, out_nd = entries processed.
//   !ALPHA (weighted sums): A += alpha w c, B += alpha w over every entry;
//          out = (bg w_bg + A) / (w_bg + B), background if that denominator
//          is not above d_min.
// Bound by instruction issue.  Two pixels per lane in scalar arithmetic, branches
// per pixel and records fetched through registers took 617 us for one 1080p view of
// 1M Gaussians, 476 this way (the whole call 992 -> 840 us); without the minimum with
// alpha_max where no opacity reaches it and with paired offsets the call went from
// 788 to 762.  Small views gain as well, though the scalar form's sub-tiles were 16x4
// (alpha-blending / weighted sums, us a call: 320x240 of 20,000 x 8 421 -> 299 / 744 -> 469,
// 640x480 of 20,000 x 10 over three decades 367 -> 255 / 288 -> 212, 160x120 of 2,048 x 8
// 389 -> 233 / 319 -> 216); packed 16x4 sub-tiles are not measured.
// ONCE: eps > 1, where the first entry that reaches a pixel is also its last, even at an
// alpha of 0, which leaves T at 1 (an instantiation of its own: the mask of such pixels
// spills at the 64 registers of the others).
template <bool ALPHA, bool ONCE = false>
__global__ void __launch_bounds__(CT, ONCE ? 24 : 32) k_gauss_blend(const ViewDesc *__restrict__ views, int n_views,
                                                    const uint32_t *__restrict__ order,
                                                    const uint2 *__restrict__ ranges,
                                                    const uint32_t *__restrict__ list,
                                                    const float4 *__restrict__ rec, BlendParams bp, float w_bg,
                                                    float *__restrict__ out_rgb, int *__restrict__ out_nd) {
    __shared__ float4 s_rec[FSTAGE][kBatchF4];
    chain_wait();
    constexpr int NR = 2, NB = batch_cells(1);
    const int lane = threadIdx.x;
    const int tile = (int)order[blockIdx.x / CSUB], sub = blockIdx.x % CSUB;
    const ViewDesc &V = views[find_view(views, n_views, tile)];
    const int local = tile - V.tile_base;
    const int tx = local % V.Tx, ty = local / V.Tx;
    const float bx0 = (float)(tx * kTile), by0 = (float)(ty * kTile + CROWS * sub);
    const int xi = tx * kTile + lane_col(lane, 0), yi = ty * kTile + CROWS * sub + lane_row(lane, 0);
    const float px = (float)xi + 0.5f, py = (float)yi + 0.5f;  // the others: 8 columns, 4 rows further
    const uint2 rg = ranges[tile];
    const float eps = fminf(bp.eps, 1.0f);  // (every pixel takes its first entry)

    // X: T (alpha; below eps: done) or B (weighted sums), of the row pairs
    float2 C0[NR], C1[NR], C2[NR], X[NR];
    int n[2 * NR];
    unsigned taken = 0u;  // ONCE: the pixels that took their entry
#pragma unroll
    for (int rr = 0; rr < NR; ++rr) {
        C0[rr] = C1[rr] = C2[rr] = make_float2(0.f, 0.f);
        const bool row = yi + 4 * rr < V.H;  // (pixels outside the image are done from the start)
        X[rr] = ALPHA ? make_float2(row && xi < V.W ? 1.f : -1.f, row && xi + 8 < V.W ? 1.f : -1.f) : make_float2(0.f, 0.f);
        n[2 * rr] = n[2 * rr + 1] = (int)(rg.y - rg.x);
    }
    CellBatches feed(list, rec + V.rec_base * kRecF4, rg.y, 1, lane);
    feed.read_ids(rg.x, 1, lane);
    feed.issue(s_rec[0], rg.x, 1, lane);
    cp_async_commit();
    feed.read_ids(rg.x + NB, 1, lane);
    int buf = 0;
    for (uint32_t base = rg.x; base < rg.y; base += NB, buf ^= 1) {
        if (ALPHA) {
            bool all = true;
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) all = all && X[rr].x < eps && X[rr].y < eps;
            if (__all_sync(0xffffffffu, all)) break;
        }
        feed.issue(s_rec[buf ^ 1], base + NB, 1, lane);  // (that buffer's batch was read in the last iteration)
        cp_async_commit();
        feed.read_ids(base + 2 * NB, 1, lane);
        cp_async_wait<1>();
        __syncwarp();
        const float4 *r = s_rec[buf];
        const bool mine = lane < feed.count(base, 1);
        const float4 rl = r[kRecF4 * lane];
        const unsigned full = __ballot_sync(0xffffffffu, mine && covers_rows(rl, bx0, by0, (float)CROWS));
        const unsigned hits = __ballot_sync(0xffffffffu, mine && touches_rows(rl, bx0, by0, (float)CROWS));
        // (batches whose opacities are all below the clamp go without the minimum, as in the
        // hybrid; not without dilation, where a flat Gaussian's L is infinite: the minimum makes
        // alpha_max of an exponent that is not a number)
        const bool clamp = bp.dilation < 1e-12f || (hits & __ballot_sync(0xffffffffu, !(r[kRecF4 * lane + 1].w < 0.9999f * bp.alpha_max))) != 0u;
        auto blend_batch = [&](auto with_clamp) {
        for (unsigned mask = hits; mask; mask &= mask - 1) {
            const int k = __ffs(mask) - 1;
            const float4 r0 = r[3 * k], r1 = r[3 * k + 1], r2 = r[3 * k + 2];
            const float2 dx = __fadd2_rn(make_float2(px, px + 8.f), make_float2(-r0.x, -r0.x));
            const float2 dy2 = __fadd2_rn(make_float2(py, py + 4.f), make_float2(-r0.y, -r0.y));
            bool h[2 * NR];  // the pixels that take the Gaussian
#pragma unroll
            for (int q = 0; q < 2 * NR; ++q) h[q] = true;
            if (!((full >> k) & 1u)) {
                const bool hx0 = fabsf(dx.x) <= r0.z, hx1 = fabsf(dx.y) <= r0.z;
#pragma unroll
                for (int rr = 0; rr < NR; ++rr) {
                    const bool hy = fabsf(rr == 0 ? dy2.x : dy2.y) <= r0.w;
                    h[2 * rr] = hx0 && hy;
                    h[2 * rr + 1] = hx1 && hy;
                }
            }
            const float2 pdx = __fmul2_rn(make_float2(r1.x, r1.x), dx);
            const float2 s2 = __fmul2_rn(make_float2(r1.z, r1.z), dy2), s22 = __fmul2_rn(s2, s2);
#pragma unroll
            for (int rr = 0; rr < NR; ++rr) {
                const float dy = rr == 0 ? dy2.x : dy2.y, q = rr == 0 ? s22.x : s22.y;
                const float2 s1 = __ffma2_rn(make_float2(r1.y, r1.y), make_float2(dy, dy), pdx);
                const float2 qd = __ffma2_rn(s1, s1, make_float2(q, q));
                float2 al = __fmul2_rn(make_float2(r1.w, r1.w), make_float2(ex2_approx(-qd.x), ex2_approx(-qd.y)));
                const bool a0 = h[2 * rr] && !(ALPHA && X[rr].x < eps) && !(ONCE && (taken >> (2 * rr) & 1u));
                const bool a1 = h[2 * rr + 1] && !(ALPHA && X[rr].y < eps) && !(ONCE && (taken >> (2 * rr) & 2u));
                if (ONCE) taken |= ((a0 ? 1u : 0u) | (a1 ? 2u : 0u)) << (2 * rr);
                if (decltype(with_clamp)::value) al = make_float2(fminf(al.x, bp.alpha_max), fminf(al.y, bp.alpha_max));
                al.x = a0 ? al.x : 0.f;
                al.y = a1 ? al.y : 0.f;
                const float2 w = __fmul2_rn(ALPHA ? X[rr] : make_float2(r2.w, r2.w), al);
                C0[rr] = __ffma2_rn(w, make_float2(r2.x, r2.x), C0[rr]);
                C1[rr] = __ffma2_rn(w, make_float2(r2.y, r2.y), C1[rr]);
                C2[rr] = __ffma2_rn(w, make_float2(r2.z, r2.z), C2[rr]);
                X[rr] = ALPHA ? __fadd2_rn(X[rr], make_float2(-w.x, -w.y)) : __fadd2_rn(X[rr], w);
                if (ALPHA && out_nd) {
                    if (a0 && (ONCE || X[rr].x < eps)) n[2 * rr] = (int)(base + k + 1 - rg.x);
                    if (a1 && (ONCE || X[rr].y < eps)) n[2 * rr + 1] = (int)(base + k + 1 - rg.x);
                }
            }
        }
        };
        if (clamp) blend_batch(std::true_type{}); else blend_batch(std::false_type{});
        __syncwarp();  // every lane is done with s_rec[buf] before it is refilled
    }
    cp_async_wait<0>();
    const long long HW = (long long)V.W * V.H;
    float *img = V.out ? V.out : out_rgb + 3 * V.pix_base;
#pragma unroll
    for (int q = 0; q < 2 * NR; ++q) {
        const int x = xi + 8 * (q & 1), y = yi + 4 * (q >> 1);
        if (!(x < V.W && y < V.H)) continue;
        const long long pin = (long long)y * V.W + x;
        const bool hi = q & 1;
        const int rr = q >> 1;
        const float Xq = hi ? X[rr].y : X[rr].x;
        float c0 = hi ? C0[rr].y : C0[rr].x, c1 = hi ? C1[rr].y : C1[rr].x, c2 = hi ? C2[rr].y : C2[rr].x;
        if (ALPHA) {
            c0 += Xq * bp.bg0; c1 += Xq * bp.bg1; c2 += Xq * bp.bg2;
            if (out_nd) out_nd[V.pix_base + pin] = n[q];
        } else {
            const float den = w_bg + Xq;
            const bool hit = den > bp.d_min;
            c0 = hit ? (bp.bg0 * w_bg + c0) / den : bp.bg0;
            c1 = hit ? (bp.bg1 * w_bg + c1) / den : bp.bg1;
            c2 = hit ? (bp.bg2 * w_bg + c2) / den : bp.bg2;
        }
        img[pin] = c0;
        img[HW + pin] = c1;
        img[2 * HW + pin] = c2;
    }
}

}  // namespace dgs

using namespace dgs;


namespace {

// The comparator's launch chain over views of one scene (caller holds ctx->mu).
dgs_status compare_chain(dgs_ctx *ctx, Workspace &ws, const Scene &sc, const std::vector<dgs_camera> &cams,
                         const dgs_compare_config &cfg, float *out_img, int *out_nd, cudaStream_t st) {
    const bool wsr = cfg.mode == DGS_COMPARE_WSR;
    const int V = (int)cams.size();
    std::vector<ViewDesc> hv;
    int tiles = 0;
    long long px = 0;
    for (int v = 0; v < V; ++v) {
        ViewDesc d = make_view(cams[v], tiles, px, 0, sc, (long long)v * sc.G, (long long)v * sc.G);
        d.N = sc.G;  // entries of this view: one per Gaussian
        d.K = 1;
        hv.push_back(d);
        tiles += d.Tx * d.Ty;
        px += (long long)cams[v].W * cams[v].H;
    }
    const long long n = (long long)V * sc.G;
    if (n >= (1LL << 32) - 1) return set_error(DGS_ERR_CAPACITY, "views x Gaussians exceeds 2^32");
    ws.V = V;
    ws.total_tiles = tiles;
    ws.total_px = px;
    ws.n_entries = n;
    ws.n_records = n;
    const long long n1 = std::max(1LL, n);
    dgs_status s;
    if ((s = ws.views.ensure(sizeof(ViewDesc) * V)) || (s = ws.small.ensure(kSmallBytes)) || (s = ws.zkey.ensure(4 * n1)) ||
        (s = ws.zval.ensure(4 * n1)) || (s = ws.rect.ensure(8 * n1)) || (s = ws.count.ensure(4 * n1)) ||
        (s = ws.offs.ensure(4 * n1)) ||
        (s = ws.scan.ensure(4 * scan_scratch_words(n1))) || (s = ensure_sort_scratch(ws, n)) ||
        (s = ws.rec.ensure(sizeof(float4) * kRecF4 * n1)) || (s = ws.ranges.ensure(8 * (size_t)std::max(1, tiles))) ||
        (s = ws.order.ensure(4 * (size_t)std::max(1, tiles))))
        return s;
    if (ws.h_views_cap < (size_t)V) {
        if (ws.h_views) cudaFreeHost(ws.h_views);
        ws.h_views = nullptr;
        ws.h_views_cap = 0;
        CK(cudaMallocHost(&ws.h_views, sizeof(ViewDesc) * V));
        ws.h_views_cap = V;
    }
    memcpy(ws.h_views, hv.data(), sizeof(ViewDesc) * V);
    CK(cudaMemcpyAsync(ws.views.p, ws.h_views, sizeof(ViewDesc) * V, cudaMemcpyHostToDevice, st));
    uint32_t *small = (uint32_t *)ws.small.p;
    CK(cudaMemsetAsync(small, 0, kSmallBytes, st));
    const ViewDesc *dv = (const ViewDesc *)ws.views.p;
    const BlendParams bp = blend_params(ctx->cfg);
    const float tau = std::isfinite(cfg.tau) && cfg.tau > 0.f ? cfg.tau : 0.f;
    launch_gauss_bin(dv, V, sc.dev(), bp, wsr, tau, (float4 *)ws.rec.p, (uint32_t *)ws.zkey.p, (uint32_t *)ws.zval.p,
                     (short4 *)ws.rect.p, (uint32_t *)ws.count.p, small + kSmallVisible, chain_prep(ws, 0, n, tiles), st);
    const uint32_t *d_vis = wsr ? nullptr : small + kSmallVisible;
    if (!wsr)  // global depth order over every visible (view, Gaussian) entry
        radix_sort_counted((uint32_t *)ws.zkey.p, (uint32_t *)ws.zval.p, n, 32, chain_sort_scratch(ws, 0), st, nullptr,
                           d_vis, false);
    // weighted sums: entries stay in index order (zval is the identity)
    launch_pair_offsets((const uint32_t *)ws.zval.p, (const uint32_t *)ws.count.p, n, nullptr, d_vis,
                        (uint32_t *)ws.offs.p, (uint32_t *)ws.scan.p, small + kSmallCounters + 8, small, kPairSlots,
                        0xFFFFFFFFu, nullptr, st);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(ws.h_small, small, 64, cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (ws.h_small[kSmallSortErr]) return set_error(DGS_ERR_TIMEOUT, "radix sort look-back wait gave up");
    const long long L = ws.h_small[kSmallTotal];
    ws.L = L;
    if ((s = ws.tkey.ensure(4 * std::max(1LL, L))) || (s = ws.tval.ensure(4 * std::max(1LL, L))) ||
        (s = ensure_sort_scratch(ws, L)))
        return s;
    int bits = 1;
    while ((1LL << bits) < tiles) ++bits;
    launch_emit((const uint32_t *)ws.offs.p, (const uint32_t *)ws.zval.p, (const short4 *)ws.rect.p, dv, V, n, n, L, tiles,
                (uint32_t *)ws.tkey.p, (uint32_t *)ws.tval.p, (bits + 7) / 8, chain_prep(ws, 1, L, 0), st, nullptr,
                d_vis, nullptr);
    sort_tiles(ws, L, bits, nullptr, st);
    launch_tile_ranges((const uint32_t *)ws.tkey.p, L, (uint2 *)ws.ranges.p, small + kSmallSortErr,
                       ws.h_small + kSmallSortErr, st);
    launch_tile_order((const uint2 *)ws.ranges.p, tiles, (uint32_t *)ws.order.p, st);
    if (tiles > 0) {
        const unsigned grid = (unsigned)tiles * CSUB;
        auto blend = [&](auto kernel, float w_bg, int *nd) {
            launch_chained(kernel, grid, CT, 0, st, dv, V, (const uint32_t *)ws.order.p, (const uint2 *)ws.ranges.p,
                           (const uint32_t *)ws.tval.p, (const float4 *)ws.rec.p, bp, w_bg, out_img, nd);
        };
        if (wsr) blend(k_gauss_blend<false>, cfg.w_bg, nullptr);
        else if (bp.eps > 1.0f) blend(k_gauss_blend<true, true>, 0.f, out_nd);
        else blend(k_gauss_blend<true>, 0.f, out_nd);
    }
    CK(cudaGetLastError());
    ws.check_flags = true;  // (a tile sort that gave up: k_tile_ranges notes it in h_small)
    return DGS_OK;
}

}  // namespace

extern "C" dgs_status dgs_render_compare(dgs_ctx *ctx, uint32_t scene_id, int32_t n_views, const uint32_t *cam_slots,
                                         const dgs_compare_config *cfg, float *out_rgb, int32_t *out_ndone,
                                         dgs_stream stream, dgs_stats *stats) {
    if (!ctx || !cfg) return set_error(DGS_ERR_INVALID_ARG, "NULL argument");
    if (n_views <= 0 || !cam_slots || !out_rgb) return set_error(DGS_ERR_INVALID_ARG, "need n_views > 0, cams, output");
    if (cfg->mode != DGS_COMPARE_ALPHA && cfg->mode != DGS_COMPARE_WSR)
        return set_error(DGS_ERR_INVALID_ARG, "unknown comparator mode");
    if (!(cfg->w_bg >= 0.f)) return set_error(DGS_ERR_INVALID_ARG, "w_bg must be >= 0");
    std::lock_guard<std::mutex> lk(ctx->mu);
    CK(cudaSetDevice(ctx->cfg.device));
    auto it = ctx->scenes.find(scene_id);
    if (it == ctx->scenes.end()) return set_error(DGS_ERR_NOT_FOUND, "unknown scene id");
    if (it->second->F > 0) return set_error(DGS_ERR_INVALID_ARG, "the comparators take explicit Gaussians");
    std::vector<dgs_camera> cams;
    for (int v = 0; v < n_views; ++v) {
        if (cam_slots[v] >= (uint32_t)kMaxCamSlots || !ctx->cam_set[cam_slots[v]])
            return set_error(DGS_ERR_NOT_FOUND, "camera slot not set");
        cams.push_back(ctx->cams[cam_slots[v]]);
    }
    cudaStream_t st = (cudaStream_t)stream;
    dgs_status s;
    std::unique_ptr<Workspace> ws = acquire_ws(ctx, st, &s);
    if (!ws) return s;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    const bool timing = stats && stats->timing;
    if (timing) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, st);
    }
    s = compare_chain(ctx, *ws, *it->second, cams, *cfg, out_rgb, out_ndone, st);
    if (timing) {
        cudaEventRecord(e1, st);
        cudaEventSynchronize(e1);
        cudaEventElapsedTime(&stats->ms_total, e0, e1);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    if (stats && !s) {
        stats->sort_length = ws->L;
        stats->num_tiles = ws->total_tiles;
        stats->visible_cells = ws->h_small[kSmallVisible];
    }
    cudaEventRecord(ws->done, st);
    ctx->pool.push_back(std::move(ws));
    return s;
}
