// Cell rasterization (Layer I, Sec. IV-B): project every ellipsoidal cell
// proxy of every view, cull it to the frustum, bound its screen footprint,
// and emit one (tile, cell) pair per covered tile.  Depth ordering comes from
// a radix sort over cells (sort.cu); a second stable sort groups by tile.
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "internal.cuh"
#include "sh.cuh"

namespace dgs {

// One thread per (view, cell).  Footprint: exact screen bounding box of the
// perspective image of the ellipsoid {c + R_Q diag(S) u, |u| <= 1}.  With the
// view-space centre c and Sigma = M M^T (M = R_view R_Q diag(S)) the planes
// X - t Z = 0 tangent to the ellipsoid solve
//   (c_z^2 - S_zz) t^2 - 2 (c_x c_z - S_xz) t + (c_x^2 - S_xx) = 0,
// whose discriminant is expanded so the c_x^2 c_z^2 terms cancel exactly.
// All of it in FP32 with a fixed operation order (see internal.cuh), so the
// tile rectangle is reproducible bit for bit.
__global__ void __launch_bounds__(256) k_cell_project(const ViewDesc *__restrict__ views, int n_views,
                                                      const SceneDev *__restrict__ scenes,
                                                      uint32_t *__restrict__ zkey, uint32_t *__restrict__ zval,
                                                      short4 *__restrict__ rect, float *__restrict__ depth,
                                                      uint32_t *__restrict__ count, uint32_t *__restrict__ visible,
                                                      float *__restrict__ vview, int flags, BinPrep prep,
                                                      const ChainSizes *__restrict__ dsz) {
    __shared__ uint32_t s_hist[4][256];  // the depth keys' digits
    for (int i = threadIdx.x; i < 4 * 256; i += blockDim.x) (&s_hist[0][0])[i] = 0u;
    __syncthreads();
    prep_clear(prep, blockIdx.x * (long long)blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
    if (dsz) n_views = dsz->n_views;
    uint32_t nvis = 0;
    for (int v = 0; v < n_views; ++v) {
    const ViewDesc &V = views[v];
    const SceneDev &SC = scenes[V.scene_slot];
    const float *__restrict__ cell = SC.cell;
    const long long N = V.N;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        const long long i = V.cell_base + n;
        float c[3];
        xform_s(V.R, V.t, cell[n], cell[N + n], cell[2 * N + n], c);
        float Rq[9], RR[9], M[9];
        rot_from_quat_s(cell[6 * N + n], cell[7 * N + n], cell[8 * N + n], cell[9 * N + n], Rq);
        const float S[3] = {cell[3 * N + n], cell[4 * N + n], cell[5 * N + n]};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                RR[3 * a + j] = fadd_s(fadd_s(fmul_s(V.R[3 * a], Rq[j]), fmul_s(V.R[3 * a + 1], Rq[3 + j])),
                                       fmul_s(V.R[3 * a + 2], Rq[6 + j]));
                M[3 * a + j] = fmul_s(RR[3 * a + j], S[j]);
            }
        auto sig = [&](int a, int b) {
            return fadd_s(fadd_s(fmul_s(M[3 * a], M[3 * b]), fmul_s(M[3 * a + 1], M[3 * b + 1])),
                          fmul_s(M[3 * a + 2], M[3 * b + 2]));
        };
        const float sxx = sig(0, 0), syy = sig(1, 1), szz = sig(2, 2), sxz = sig(0, 2), syz = sig(1, 2);
        float dz = c[2];  // the sort depth
        short4 r = make_short4(-1, -1, -1, -1);
        bool vis = fsub_s(c[2], fsqrt_s(szz)) > V.znear;
        if (!vis && (flags & DGS_FLAG_NEAR_FULL) && fadd_s(c[2], fsqrt_s(szz)) > V.znear) {
            // straddles the near plane: conservatively every tile, nearest first
            vis = true;
            dz = c[2] > 0.0f ? c[2] : 0.0f;
            r = make_short4(0, 0, (short)(V.Tx - 1), (short)(V.Ty - 1));
        } else if (vis) {
            const float czz = fmul_s(c[2], c[2]);
            const float a = fsub_s(czz, szz);
            float lo[2], hi[2];
#pragma unroll
            for (int ax = 0; ax < 2; ++ax) {
                const float cu = c[ax];
                const float suu = ax == 0 ? sxx : syy, suz = ax == 0 ? sxz : syz;
                const float f = ax == 0 ? V.fx : V.fy, pp = ax == 0 ? V.cx : V.cy;
                const float cuz = fmul_s(cu, c[2]), cuu = fmul_s(cu, cu);
                const float b = fsub_s(cuz, suz);
                float disc = fsub_s(fadd_s(fsub_s(fmul_s(czz, suu), fmul_s(fmul_s(2.0f, cuz), suz)), fmul_s(cuu, szz)),
                                    fsub_s(fmul_s(suu, szz), fmul_s(suz, suz)));
                disc = fmaxf(disc, 0.0f);
                const float sq = fsqrt_s(disc);
                lo[ax] = fadd_s(fmul_s(f, fdiv_s(fsub_s(b, sq), a)), pp);
                hi[ax] = fadd_s(fmul_s(f, fdiv_s(fadd_s(b, sq), a)), pp);
            }
            const float fW = (float)V.W, fH = (float)V.H;
            vis = hi[0] >= 0.0f && lo[0] < fW && hi[1] >= 0.0f && lo[1] < fH;
            if (vis) {
                const float ft = (float)kTile;
                int tx0 = (int)floorf(fdiv_s(fmaxf(lo[0], 0.0f), ft));
                int ty0 = (int)floorf(fdiv_s(fmaxf(lo[1], 0.0f), ft));
                int tx1 = (int)floorf(fdiv_s(fminf(hi[0], fW), ft));
                int ty1 = (int)floorf(fdiv_s(fminf(hi[1], fH), ft));
                tx1 = min(tx1, V.Tx - 1);
                ty1 = min(ty1, V.Ty - 1);
                r = make_short4((short)tx0, (short)ty0, (short)tx1, (short)ty1);
            }
        }
        rect[i] = r;
        depth[i] = dz;
        // v_n of this view (Sec. V-A): the scalar, or clamp(sum_lm k_lm Y_lm(d), 0, 1)
        // with d the unit vector from the eye to the cell centre
        float vn = cell[10 * N + n];
        if (SC.vsh) {
            float d0 = cell[n] - V.eye[0], d1 = cell[N + n] - V.eye[1], d2 = cell[2 * N + n] - V.eye[2];
            const float il = rsqrtf(d0 * d0 + d1 * d1 + d2 * d2);
            d0 *= il; d1 *= il; d2 *= il;
            float Y[16];
            sh_eval(d0, d1, d2, SC.v_sh_degree, Y);
            const int Cv = (SC.v_sh_degree + 1) * (SC.v_sh_degree + 1);
            float raw = 0.f;
            for (int c = 0; c < Cv; ++c) raw += SC.vsh[c * N + n] * Y[c];
            vn = fminf(fmaxf(raw, 0.f), 1.f);
        }
        vview[i] = vn;
        // depth key: positive float bits order like the floats; culled last
        const uint32_t key = vis ? __float_as_uint(dz) : 0xFFFFFFFFu;
        zkey[i] = key;
        zval[i] = (uint32_t)i;
        count[i] = vis ? (uint32_t)((r.z - r.x + 1) * (r.w - r.y + 1)) : 0u;
        nvis += vis ? 1u : 0u;
        if (vis) {
#pragma unroll
            for (int p = 0; p < 4; ++p) atomicAdd(&s_hist[p][(key >> (8 * p)) & 255u], 1u);
        }
    }
    }
    // one atomic per warp for the visible-cell statistic
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nvis += __shfl_xor_sync(0xffffffffu, nvis, o);
    if ((threadIdx.x & 31) == 0 && nvis) atomicAdd(visible, nvis);
    __syncthreads();
    for (int i = threadIdx.x; i < 4 * 256; i += blockDim.x) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(prep.hist + i, c);
    }
}

static int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    const long long cap = 152LL * 32;  // 152 SMs x resident blocks; grid-stride beyond
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

void launch_cell_project(const ViewDesc *views, int n_views, const SceneDev *scenes, long long n_entries,
                         uint32_t *zkey, uint32_t *zval, short4 *rect, float *depth, uint32_t *count,
                         uint32_t *visible, float *vview, int flags, const BinPrep &prep, cudaStream_t st,
                         const ChainSizes *dsz) {
    // eight blocks an SM at most: each adds its digit counts to the global ones once
    k_cell_project<<<std::min(grid_for(n_entries / n_views + 1, 256), 152 * 8), 256, 0, st>>>(
        views, n_views, scenes, zkey, zval, rect, depth, count, visible, vview, flags, prep, dsz);
}

// Output slot j belongs to the last entry e with offs[e] <= j.  A block takes
// runs of EM_TB consecutive slots.  Two warps find the run's first and last owners
// in global memory, 32 probes at a time (four dependent reads for a million
// entries; one thread's two binary searches were 40, most of a small view's 19 us
// in here).  When at most EM_TB entries lie between them (always for the
// depth-sorted entries, of which each owns a slot) their offsets are staged in
// shared memory with their first tile, row lengths and cell, otherwise
// (entries that own no slot interleaved, as in the weighted-sum comparator's index
// order) they are searched in global memory.  A thread finds the owner of the first
// of its eight consecutive slots and walks on from there, with one division for the
// first slot's tile, and writes the eight keys and cells as vectors.
// Entries are in depth order, so the emitted sequence is (depth, cell)-ordered
// within every tile; the stable tile sort keeps that order.  The keys' digits are
// counted on the way, runs of equal digits of a thread at once.
constexpr int EM_THREADS = 256, EM_ITEMS = 8, EM_TB = EM_THREADS * EM_ITEMS;

// Last entry e in [0, n) with offs[e] <= j (0 if there is none), by one warp.
__device__ __forceinline__ long long warp_owner(const uint32_t *__restrict__ offs, long long n, long long j, int lane) {
    long long lo = 0, hi = n;  // offs[lo] <= j (or lo = 0), offs[hi] > j (or hi = n)
    while (hi - lo > 1) {
        const long long step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step;  // probes above lo
        const bool le = at < hi && (long long)offs[at] <= j;
        const int m = __popc(__ballot_sync(0xffffffffu, le));  // (offs is sorted: the first m probes)
        const long long nlo = lo + m * step;
        hi = min(hi, nlo + step);
        lo = nlo;
    }
    return lo;
}

__global__ void __launch_bounds__(EM_THREADS) k_emit(const uint32_t *__restrict__ offs,
                                                     const uint32_t *__restrict__ zval,
                                                     const short4 *__restrict__ rect,
                                                     const ViewDesc *__restrict__ views, int n_views,
                                                     long long n_entries, long long n_all, long long L, int n_tiles,
                                                     uint32_t *__restrict__ tkey, uint32_t *__restrict__ tval,
                                                     int passes, BinPrep prep, const ChainSizes *__restrict__ dsz,
                                                     const uint32_t *__restrict__ d_n,
                                                     const uint32_t *__restrict__ d_L) {
    // the run's entries: first slot (less j0), first tile, tiles per row | tiles of the
    // view's row << 16, cell
    __shared__ int s_off[EM_TB];
    __shared__ uint32_t s_tile[EM_TB], s_wt[EM_TB], s_cell[EM_TB];
    __shared__ uint32_t s_hist[4][256];
    __shared__ long long s_own[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < passes * 256; i += EM_THREADS) (&s_hist[0][0])[i] = 0u;
    chain_wait();
    prep_clear(prep, blockIdx.x * (long long)EM_THREADS + tid, (long long)gridDim.x * EM_THREADS);
    if (dsz) {
        n_views = dsz->n_views;
        n_all = dsz->n_entries;
        n_tiles = dsz->total_tiles;
    }
    if (d_n) n_entries = *d_n;
    if (d_L) L = *d_L;
    // (bounds: only a sort that gave up can leave an entry outside the arrays)
    auto entry = [&](long long e, uint32_t &tile, uint32_t &wt, uint32_t &cell) {
        const uint32_t vi = (uint32_t)min((long long)zval[e], n_all - 1);
        int vlo = 0, vhi = n_views;  // view owning entry vi
        while (vhi - vlo > 1) {
            const int mid = (vlo + vhi) >> 1;
            if (views[mid].cell_base <= (long long)vi) vlo = mid; else vhi = mid;
        }
        const ViewDesc &V = views[vlo];
        const short4 r = rect[vi];
        tile = (uint32_t)(V.tile_base + r.y * V.Tx + r.x);
        wt = (uint32_t)(r.z - r.x + 1) | (uint32_t)V.Tx << 16;
        cell = (uint32_t)((long long)vi - V.cell_base);
    };
    for (long long j0 = blockIdx.x * (long long)EM_TB; j0 < L; j0 += (long long)gridDim.x * EM_TB) {
        const int run = (int)min((long long)EM_TB, L - j0);  // slots [j0, j0 + run)
        __syncthreads();  // the last run's entries are read (and s_hist is clear)
        if (warp < 2) {
            const long long o = warp_owner(offs, n_entries, warp == 0 ? j0 : j0 + run - 1, lane);
            if (lane == 0) s_own[warp] = o;
        }
        __syncthreads();
        const long long e0 = s_own[0];
        const int ne = (int)min(s_own[1] - e0 + 1, (long long)INT_MAX);  // the run's owners are entries [e0, e0 + ne)
        const bool staged = ne <= EM_TB;
        if (staged)
            for (int i = tid; i < ne; i += EM_THREADS) {
                s_off[i] = (int)((long long)offs[e0 + i] - j0);
                entry(e0 + i, s_tile[i], s_wt[i], s_cell[i]);
            }
        __syncthreads();
        const int js = tid * EM_ITEMS;
        if (js >= run) continue;
        auto off = [&](int i) { return staged ? s_off[i] : (int)((long long)offs[e0 + i] - j0); };
        int own = 0, hi = ne;  // last i in [0, ne) with off(i) <= js
        while (hi - own > 1) {
            const int mid = (own + hi) >> 1;
            if (off(mid) <= js) own = mid; else hi = mid;
        }
        uint32_t key[EM_ITEMS], cell[EM_ITEMS];
        uint32_t tile = 0, wt = 1, cellid = 0;  // of the current owner
        int next = js, x = 0;                   // its slots end before `next`; the slot's column
        const long long j = j0 + js, j1 = j0 + run;
#pragma unroll
        for (int i = 0; i < EM_ITEMS; ++i) {
            key[i] = cell[i] = 0u;
            if (js + i < run) {
                if (js + i >= next) {  // enter the owner of this slot
                    if (i > 0)
                        while (own + 1 < ne && off(own + 1) <= js + i) ++own;
                    if (staged) {
                        tile = s_tile[own];
                        wt = s_wt[own];
                        cellid = s_cell[own];
                    } else {
                        entry(e0 + own, tile, wt, cellid);
                    }
                    x = 0;  // (an owner entered past the thread's first slot is entered at its first)
                    if (i == 0) {
                        const uint32_t local = (uint32_t)(js - off(own)), y = local / (wt & 0xffffu);
                        x = (int)(local - y * (wt & 0xffffu));
                        tile += y * (wt >> 16);
                    }
                    next = own + 1 < ne ? off(own + 1) : run;
                }
                key[i] = min(tile + (uint32_t)x, (uint32_t)(n_tiles - 1));
                cell[i] = cellid;
                if (++x == (int)(wt & 0xffffu)) {
                    x = 0;
                    tile += wt >> 16;
                }
            }
        }
        if (j + EM_ITEMS <= j1) {
#pragma unroll
            for (int i = 0; i < EM_ITEMS; i += 4) {
                *reinterpret_cast<uint4 *>(tkey + j + i) = make_uint4(key[i], key[i + 1], key[i + 2], key[i + 3]);
                *reinterpret_cast<uint4 *>(tval + j + i) = make_uint4(cell[i], cell[i + 1], cell[i + 2], cell[i + 3]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < EM_ITEMS; ++i)
                if (j + i < j1) {
                    tkey[j + i] = key[i];
                    tval[j + i] = cell[i];
                }
        }
        const int n = (int)min((long long)EM_ITEMS, j1 - j);
        for (int p = 0; p < passes; ++p) {
            uint32_t d = (key[0] >> (8 * p)) & 255u, run = 1;
#pragma unroll
            for (int i = 1; i < EM_ITEMS; ++i) {
                const uint32_t di = (key[i] >> (8 * p)) & 255u;
                if (i < n) {
                    if (di != d) {
                        atomicAdd(&s_hist[p][d], run);
                        d = di;
                        run = 0;
                    }
                    ++run;
                }
            }
            atomicAdd(&s_hist[p][d], run);
        }
    }
    __syncthreads();
    for (int i = tid; i < passes * 256; i += EM_THREADS) {
        const uint32_t c = (&s_hist[0][0])[i];
        if (c) atomicAdd(prep.hist + i, c);
    }
}

void launch_emit(const uint32_t *offs, const uint32_t *zval_sorted, const short4 *rect, const ViewDesc *views,
                 int n_views, long long n_entries, long long n_all, long long L, int n_tiles, uint32_t *tkey,
                 uint32_t *tval, int passes, const BinPrep &prep, cudaStream_t st, const ChainSizes *dsz,
                 const uint32_t *d_n, const uint32_t *d_L) {
    if (L == 0) return;
    // eight blocks an SM at most: each adds its digit counts to the global ones once
    const long long runs = (L + EM_TB - 1) / EM_TB;
    launch_chained(k_emit, (unsigned)std::min<long long>(runs, 152 * 8), EM_THREADS, 0, st,
        offs, zval_sorted, rect, views, n_views, n_entries, n_all, L, n_tiles, tkey, tval, passes, prep, dsz, d_n, d_L);
}

// [start, end) of every non-empty tile from the tile-sorted keys; empty
// tiles keep the (0,0) the caller cleared them to -- and all tiles do if a wait of
// the chain's sorts or of its scan gave up: slots that no pass wrote hold whatever
// the buffer held, keys beyond the last tile and cells beyond the last cell.  With
// empty lists no later kernel reads them.
__global__ void k_tile_ranges(const uint32_t *__restrict__ key, long long L, const uint32_t *__restrict__ d_L,
                              uint2 *__restrict__ ranges, const uint32_t *__restrict__ err,
                              uint32_t *__restrict__ host_err) {
    chain_wait();
    const uint32_t gave_up = *err;  // (requested together with the count)
    if (d_L) L = *d_L;
    if (gave_up) {
        if (host_err && blockIdx.x == 0 && threadIdx.x == 0) *host_err = 1u;
        return;
    }
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < L; j += (long long)gridDim.x * blockDim.x) {
        const uint32_t k = key[j];
        if (j == 0 || key[j - 1] != k) ranges[k].x = (uint32_t)j;
        if (j == L - 1 || key[j + 1] != k) ranges[k].y = (uint32_t)(j + 1);
    }
}

void launch_tile_ranges(const uint32_t *tkey_sorted, long long L, uint2 *ranges, const uint32_t *err, uint32_t *host_err,
                        cudaStream_t st, const uint32_t *d_L) {
    if (L == 0) return;
    launch_chained(k_tile_ranges, grid_for(L, 256), 256, 0, st, tkey_sorted, L, d_L, ranges, err, host_err);
}

// Tiles by descending list length (in steps of a quarter of a power of two), for
// the blend kernels' launch order: a tile's blend takes as long as its list, and a
// long one started last would leave the chip idle but for it.  One cluster counts
// the lengths in each CTA's shared memory, adds the counts up over distributed shared
// memory and places its tiles (one CTA up to TO_SINGLE tiles, where a cluster's
// barriers would cost more than it saves; 4K views have 32,400).  The order within a
// step is that of the atomics; no result depends on it.
constexpr int TO_THREADS = 1024, TO_ITEMS = 4, TO_CTAS = 8, TO_SINGLE = 4096;
__device__ __forceinline__ int length_step(uint2 r) {  // 0 the longest, 127 the empty lists
    const uint32_t len = r.y - r.x;
    if (len == 0u) return 127;
    const int e = 31 - __clz(len);
    return 126 - min(126, 4 * e + (int)(((unsigned long long)len << 2 >> e) & 3u));
}
__global__ void __launch_bounds__(TO_THREADS) k_tile_order(const uint2 *__restrict__ ranges, int n_tiles,
                                                           uint32_t *__restrict__ order,
                                                           const ChainSizes *__restrict__ dsz) {
    __shared__ uint32_t s_cnt[128], s_at[128], s_warp[4];
    const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
    const int tid = threadIdx.x;
    if (tid < 128) s_cnt[tid] = 0u;
    __syncthreads();
    chain_wait();
    if (dsz) n_tiles = dsz->total_tiles;
    const int stride = ctas * TO_THREADS;
    auto sweep = [&](auto &&f) {
        for (int t0 = rank * TO_THREADS + tid; t0 < n_tiles; t0 += stride * TO_ITEMS) {
            uint2 r[TO_ITEMS];
#pragma unroll
            for (int i = 0; i < TO_ITEMS; ++i)
                if (t0 + i * stride < n_tiles) r[i] = ranges[t0 + i * stride];
#pragma unroll
            for (int i = 0; i < TO_ITEMS; ++i)
                if (t0 + i * stride < n_tiles) f(t0 + i * stride, length_step(r[i]));
        }
    };
    sweep([&](int, int step) { atomicAdd(&s_cnt[step], 1u); });
    cl.sync();
    uint32_t all = 0u, before = 0u, x = 0u;
    if (tid < 128) {  // step tid: its tiles in all CTAs and in those before this one
        for (int q = 0; q < ctas; ++q) {
            const uint32_t c = *cl.map_shared_rank(&s_cnt[tid], q);
            all += c;
            before += q < rank ? c : 0u;
        }
        x = all;  // inclusive sum over the steps
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if ((tid & 31) >= o) x += y;
        }
        if ((tid & 31) == 31) s_warp[tid >> 5] = x;
    }
    __syncthreads();
    if (tid < 128) {
        for (int w = 0; w < (tid >> 5); ++w) x += s_warp[w];
        s_at[tid] = x - all + before;
    }
    cl.sync();  // (no CTA leaves, or reads s_at, before all counts are read)
    sweep([&](int t, int step) { order[atomicAdd(&s_at[step], 1u)] = (uint32_t)t; });
}

void launch_tile_order(const uint2 *ranges, int n_tiles, uint32_t *order, cudaStream_t st, const ChainSizes *dsz) {
    if (n_tiles == 0) return;
    const unsigned ctas = n_tiles <= TO_SINGLE ? 1 : TO_CTAS;
    launch_chained(k_tile_order, ctas, TO_THREADS, 0, st, ClusterSize{ctas}, ranges, n_tiles, order, dsz);
}

}  // namespace dgs
