// Stable LSD radix sort of (uint32 key, uint32 value) pairs, 8-bit digits,
// one "onesweep" pass per digit: every CTA ranks a partition (3072 items, or 1024 in
// small sorts) locally, reorders it by digit in shared memory, learns the global
// offset of each digit from its predecessors through decoupled look-back (Merrill &
// Garland single-pass prefix scan, applied per digit as in Adinets & Merrill's
// Onesweep), and writes coalesced runs.  The digit counts of all passes are there
// beforehand: a render's kernels count the keys that they write (BinPrep), and
// radix_sort_pairs reads its keys once for them.
//
// Sec. IV-B sorts the cell sequence with a radix sort; its cost grows with
// the sequence length, which is why the sort runs over cells, not Gaussians
// (Sec. VII-D, Tab. VI).
//
// Every wait on another CTA is bounded: after kSpinLimit polls the CTA sets
// *err, treats the missing count as 0 and carries on, so the kernel always
// finishes; the host turns a set flag into an error.
#include <algorithm>

#include "internal.cuh"

namespace dgs {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
// Items per thread.  A partition of 3072 items streams best; up to
// kSmallSort items, where a pass is one partition's latency and not its
// rate (a lone 3072-item partition ranks twelve items a thread one after
// another), partitions of 1024 spread them over more CTAs (four passes over 100,000
// keys 39 -> 32 us, over 200,000 41 -> 36; over 800,000 nothing is gained).
constexpr int RS_ITEMS = 12, RS_ITEMS_SMALL = 4;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;      // 3072 items per partition
constexpr int RS_TILE_SMALL = RS_THREADS * RS_ITEMS_SMALL;
constexpr long long kSmallSort = 262144;
static_assert(RS_TILE == kSortPartition, "the partition size is shared with the fixed scratch of sort_noalloc.cu");
static_assert(kSmallSort / RS_TILE_SMALL <= (1 << 20) / RS_TILE, "small partitions fit that scratch's look-back words");
constexpr uint32_t FLAG_AGG = 1u << 30;             // partition's own count published
constexpr uint32_t FLAG_INC = 2u << 30;             // inclusive prefix published
constexpr uint32_t COUNT_MASK = (1u << 30) - 1;
constexpr int kSpinLimit = 1 << 22;

// Fault injection for the failure-detection tests (dgs_debug_inject_fault,
// DGS_FAULT_SORT_WAIT): while set to kFaultSort, partition 0 of a sort never
// publishes its digit counts (kFaultScan: that of a pair-offset scan its sum) and a wait
// gives up after kFaultSpinLimit polls, so the look-back waits of the other
// partitions run out -- each one still bounded.
//
// After a wait that gave up: the missing partition counts as 0, so that
// pass's destinations stay below their digits' true ends, but some slots are not
// written.  The next pass reads there whatever the buffer held, keys that are in no
// digit count, and a digit can then run past its end: a partition with a digit that would
// run past the arrays is not written (k_rs_pass).  The kernels of a chain that read what the sorts
// left take it through a bound (k_pair_offsets, k_emit, k_decode_samples) or, from
// the tile ranges on, not at all: k_tile_ranges leaves every tile's list empty.
__device__ int g_rs_fault = 0;
constexpr int kFaultSort = 1, kFaultScan = 2;
constexpr int kFaultSpinLimit = 1024;

cudaError_t set_sort_fault(int which) { return cudaMemcpyToSymbol(g_rs_fault, &which, sizeof(int)); }

// partitions that the scratch of a sort of up to n items is sized for
long long sort_parts_for(long long n) {
    return std::max((n + RS_TILE - 1) / RS_TILE, (std::min(n, kSmallSort) + RS_TILE_SMALL - 1) / RS_TILE_SMALL);
}

// Histograms of every digit of every pass in one read of the keys.
// Also clears the look-back words of the first pass (`words` at status0).
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint32_t *__restrict__ keys, long long n, int passes,
                                                        uint32_t *__restrict__ hist, uint32_t *__restrict__ status0,
                                                        long long words) {
    for (long long i = blockIdx.x * (long long)RS_THREADS + threadIdx.x; i < words; i += (long long)gridDim.x * RS_THREADS)
        status0[i] = 0u;
    __shared__ uint32_t sh[4][256];
    for (int i = threadIdx.x; i < 4 * 256; i += RS_THREADS) (&sh[0][0])[i] = 0;
    __syncthreads();
    for (long long i = blockIdx.x * (long long)RS_THREADS + threadIdx.x; i < n; i += (long long)gridDim.x * RS_THREADS) {
        const uint32_t k = keys[i];
        for (int p = 0; p < passes; ++p) atomicAdd(&sh[p][(k >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += RS_THREADS) {
        const uint32_t c = (&sh[0][0])[i];
        if (c) atomicAdd(&hist[i], c);
    }
}

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t *p) { return *(const volatile uint32_t *)p; }

// Pass `pass` of the sort.  The data ping-pongs between (k0, v0) and
// (k1, v1).  hist: the digits' counts.  With skip_trivial, a pass whose digit is
// 0 for every key (the histogram says so) is the identity permutation and does
// nothing; every pass then takes its input from the buffer the previous
// non-trivial pass wrote, and the look-back arrays alternate over non-trivial
// passes.  With d_live, pass 0 leaves out the items whose key is 0xFFFFFFFF (they are
// not in the histograms), *d_live stay, and later passes sort those; no pass is
// skipped then (a skipped first pass would leave nothing out).
__device__ __forceinline__ bool rs_trivial(const uint32_t *hist, int q, long long n) {
    return (long long)hist[256 * q] == n;
}

constexpr int RS_LOOK = 8;  // predecessors that a look-back reads at a time

// A pass is latency more than rate: 5.6M pairs move 90 MB, 13 us at the copy rate, and
// take 52 (61 with the values held in registers from the start and the look-back
// before the reordering, 80 registers and three CTAs an SM; four at 64).

template <int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 4) k_rs_pass(uint32_t *__restrict__ k0, uint32_t *__restrict__ v0,
                                                        uint32_t *__restrict__ k1, uint32_t *__restrict__ v1,
                                                        long long n, const uint32_t *__restrict__ d_n,
                                                        const uint32_t *__restrict__ d_live, int pass,
                                                        const uint32_t *__restrict__ hist, bool skip_trivial,
                                                        uint32_t *__restrict__ status0, uint32_t *__restrict__ status1,
                                                        uint32_t *__restrict__ counter,
                                                        uint32_t *__restrict__ err) {
    constexpr int TILE = RS_THREADS * ITEMS, WARP_ITEMS = 32 * ITEMS;
    __shared__ uint32_t s_warp[RS_WARPS][256];   // per-warp digit counts, then per-warp offsets
    __shared__ uint32_t s_base[256];             // global destination of the partition's first item per digit
    __shared__ uint32_t s_local[256];            // partition-local start of each digit
    __shared__ uint32_t s_wsum[RS_WARPS];
    __shared__ uint32_t s_key[TILE], s_val[TILE];  // the partition in digit order
    __shared__ uint32_t s_part, s_cnt;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_wait();
    if (d_n) n = *d_n;
    const bool drop = d_live && pass == 0;
    if (d_live && pass > 0) n = *d_live;
    int ord = pass;  // non-trivial passes before this one
    if (skip_trivial) {
        if (rs_trivial(hist, pass, n)) return;
        ord = 0;
        for (int q = 0; q < pass; ++q) ord += rs_trivial(hist, q, n) ? 0 : 1;
    }
    const int shift = 8 * pass;
    const uint32_t *__restrict__ kin = (ord & 1) ? k1 : k0;
    const uint32_t *__restrict__ vin = (ord & 1) ? v1 : v0;
    uint32_t *__restrict__ kout = (ord & 1) ? k0 : k1;
    uint32_t *__restrict__ vout = (ord & 1) ? v0 : v1;
    uint32_t *__restrict__ status = (ord & 1) ? status1 : status0;
    uint32_t *__restrict__ status_next = (ord & 1) ? status0 : status1;
    const long long n_parts = (n + TILE - 1) / TILE;
    if (blockIdx.x >= n_parts) return;  // the first min(grid, n_parts) CTAs take every partition
    // exclusive scan over the 256 threads (every CTA scans the 256 counts for itself)
    auto scan256 = [&](uint32_t c) {
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_wsum[warp] = x;
        __syncthreads();
        uint32_t wb = 0;
        for (int w = 0; w < warp; ++w) wb += s_wsum[w];
        return wb + x - c;
    };
    const uint32_t digit_base = scan256(hist[256 * pass + tid]);  // of digit tid
    // Persistent CTAs claim partitions in increasing order: a partition only
    // waits for earlier ones, which CTAs that are already running own.
    for (;;) {
        __syncthreads();
        if (tid == 0) s_part = atomicAdd(counter, 1u);
        for (int i = tid; i < RS_WARPS * 256; i += RS_THREADS) (&s_warp[0][0])[i] = 0;
        __syncthreads();
        const long long part = s_part;
        if (part >= n_parts) break;
        // the next pass's look-back words of this partition: that array was
        // last used by the previous pass, which has finished
        status_next[part * 256 + tid] = 0u;
        const long long base = part * TILE + (long long)warp * WARP_ITEMS;

        uint32_t key[ITEMS], rank[ITEMS];
        unsigned live = 0;  // bit `it`: the item is there
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const long long idx = base + it * 32 + lane;
            const bool ok = idx < n;
            key[it] = ok ? kin[idx] : 0u;
            live |= ok && !(drop && key[it] == 0xFFFFFFFFu) ? 1u << it : 0u;
        }
        const unsigned lt_mask = (1u << lane) - 1u;
        // rank inside the warp, in item order (it, lane): stable.  The lanes with an
        // equal digit come from one ballot per bit: independent of one another and
        // of the other items', where match.any is a serial instruction.
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const bool ok = (live >> it) & 1u;
            unsigned peers = __ballot_sync(0xffffffffu, ok);
            const uint32_t d = (key[it] >> shift) & 255u;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const bool bit = (d >> b) & 1u;
                const unsigned m = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? m : ~m;
            }
            rank[it] = peers;
        }
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const bool ok = (live >> it) & 1u;
            const unsigned peers = rank[it];
            const uint32_t d = (key[it] >> shift) & 255u;
            const uint32_t before = s_warp[warp][d];
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1) s_warp[warp][d] = before + __popc(peers);
            rank[it] = before + __popc(peers & lt_mask);
            __syncwarp();
        }
        __syncthreads();
        // thread t owns digit t: partition total and per-warp exclusive offsets
        const int d = tid;
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t c = s_warp[w][d];
            s_warp[w][d] = total;
            total += c;
        }
        uint32_t *my = status + part * 256 + d;
        const bool fault = g_rs_fault == kFaultSort;
        if (part == 0) {
            if (!fault) atomicExch(my, FLAG_INC | total);
        } else {
            atomicExch(my, FLAG_AGG | total);
        }
        s_local[d] = scan256(total);  // partition-local digit starts
        if (d == 255) s_cnt = s_local[255] + total;
        __syncthreads();
        // the partition in digit order in shared memory (which frees the registers and
        // gives the predecessors time before the look-back)
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            if ((live >> it) & 1u) {
                const uint32_t dg = (key[it] >> shift) & 255u;
                const uint32_t lp = s_local[dg] + s_warp[warp][dg] + rank[it];
                s_key[lp] = key[it];
                s_val[lp] = vin[base + it * 32 + lane];
            }
        }
        if (part == 0) {
            s_base[d] = digit_base;
        } else {
            // RS_LOOK predecessors' words are requested together: a look-back over p
            // partitions costs p / RS_LOOK memory latencies
            const int limit = fault ? kFaultSpinLimit : kSpinLimit;
            uint32_t excl = 0;
            bool found = false;
            for (long long p = part - 1; p >= 0 && !found; p -= RS_LOOK) {
                uint32_t w[RS_LOOK];
#pragma unroll
                for (int i = 0; i < RS_LOOK; ++i) w[i] = p - i >= 0 ? ld_volatile(status + (p - i) * 256 + d) : FLAG_INC;
#pragma unroll
                for (int i = 0; i < RS_LOOK; ++i) {
                    if (found) break;
                    uint32_t s = w[i];
                    int spins = 0;
                    while ((s & (FLAG_AGG | FLAG_INC)) == 0u) {
                        if (++spins > limit) { atomicOr(err, 1u); s = FLAG_INC; break; }
                        __nanosleep(64);
                        s = ld_volatile(status + (p - i) * 256 + d);
                    }
                    excl += s & COUNT_MASK;
                    found = (s & FLAG_INC) != 0u;
                }
            }
            atomicExch(my, FLAG_INC | (excl + total));
            s_base[d] = digit_base + excl;
        }
        // a digit that would run past the arrays (only after a wait that gave up): nothing is
        // written (one test per digit: per item it costs a comparator view of 1M Gaussians 4 us of 770)
        const bool past = __syncthreads_or(s_base[d] + total > (uint32_t)n);
        // out with consecutive threads on consecutive destinations within each digit
        const int cnt = past ? 0 : (int)s_cnt;
        for (int i = tid; i < cnt; i += RS_THREADS) {
            const uint32_t k = s_key[i], dg = (k >> shift) & 255u;
            const uint32_t dst = s_base[dg] + ((uint32_t)i - s_local[dg]);
            kout[dst] = k;
            vout[dst] = s_val[i];
        }
    }
}

// Copy the result back to (kd, vd) if an odd number of non-trivial passes
// left it in (ks, vs).
__global__ void k_copy_pairs(const uint32_t *__restrict__ ks, const uint32_t *__restrict__ vs, uint32_t *__restrict__ kd,
                             uint32_t *__restrict__ vd, long long n, const uint32_t *__restrict__ d_n,
                             const uint32_t *__restrict__ hist, int passes) {
    if (d_n) n = *d_n;
    int ord = 0;
    for (int q = 0; q < passes; ++q) ord += rs_trivial(hist, q, n) ? 0 : 1;
    if (!(ord & 1)) return;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        kd[i] = ks[i];
        vd[i] = vs[i];
    }
}

// The passes of a sort whose histograms and cleared look-back words are in place.
// Returns whether the result sits in the alternate buffers (a device-counted
// sort that skips trivial passes copies it back itself).
static bool radix_passes(uint32_t *keys, uint32_t *vals, long long n, int passes, const SortScratch &s, cudaStream_t st,
                         const uint32_t *d_n, const uint32_t *d_live, bool skip) {
    const bool small = n <= kSmallSort;
    const long long tile = small ? RS_TILE_SMALL : RS_TILE, parts = (n + tile - 1) / tile;
    // look-back words: two arrays of 256 per partition, used by alternate passes
    uint32_t *status[2] = {s.status, s.status + 256 * parts};
    // persistent grid: the CTAs that every SM of the current device holds at once
    const void *kernel = small ? (const void *)k_rs_pass<RS_ITEMS_SMALL> : (const void *)k_rs_pass<RS_ITEMS>;
    const unsigned grid = (unsigned)std::min(parts, resident_ctas(kernel, RS_THREADS));
    for (int p = 0; p < passes; ++p) {
        if (small)
            launch_chained(k_rs_pass<RS_ITEMS_SMALL>, grid, RS_THREADS, 0, st, keys, vals, s.keys_alt, s.vals_alt, n, d_n,
                           d_live, p, s.hist, skip, status[0], status[1], s.counters + p, s.err);
        else
            launch_chained(k_rs_pass<RS_ITEMS>, grid, RS_THREADS, 0, st, keys, vals, s.keys_alt, s.vals_alt, n, d_n, d_live, p,
                           s.hist, skip, status[0], status[1], s.counters + p, s.err);
    }
    if (!skip) return passes & 1;
    k_copy_pairs<<<152 * 2, 256, 0, st>>>(s.keys_alt, s.vals_alt, keys, vals, n, d_n, s.hist, passes);
    return false;
}

long long sort_status_words(long long n) {
    const long long tile = n <= kSmallSort ? RS_TILE_SMALL : RS_TILE;
    return 256 * ((n + tile - 1) / tile);
}

bool radix_sort_counted(uint32_t *keys, uint32_t *vals, long long n, int bits, const SortScratch &s, cudaStream_t st,
                        const uint32_t *d_n, const uint32_t *d_live, bool skip_trivial) {
    if (n <= 0 || bits <= 0) return false;
    return radix_passes(keys, vals, n, (bits + 7) / 8, s, st, d_n, d_live, skip_trivial && !d_live);
}

int radix_sort_pairs(uint32_t *keys, uint32_t *vals, long long n, int bits, const SortScratch &s, cudaStream_t st) {
    if (n <= 1 || bits <= 0) return 0;
    const int passes = (bits + 7) / 8;
    cudaMemsetAsync(s.hist, 0, sizeof(uint32_t) * 4 * 256, st);
    cudaMemsetAsync(s.counters, 0, sizeof(uint32_t) * 4, st);
    int hb = (int)((n + RS_THREADS * 8 - 1) / (RS_THREADS * 8));
    if (hb > 152 * 8) hb = 152 * 8;
    k_rs_hist<<<hb, RS_THREADS, 0, st>>>(keys, n, passes, s.hist, s.status, sort_status_words(n));
    if (radix_passes(keys, vals, n, passes, s, st, nullptr, nullptr, false)) {
        cudaMemcpyAsync(keys, s.keys_alt, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
        cudaMemcpyAsync(vals, s.vals_alt, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
    }
    return passes;
}

// ---------------------------------------------------------------- offsets of the entries' pairs
// Exclusive scan of the sorted entries' tile counts, count[idx[i]], in one pass:
// each 2048-entry partition publishes its sum and takes its predecessors' by
// decoupled look-back, one warp reading 32 of them at a time (words: value and
// flag in 64 bits; partitions are claimed in order, waits are bounded as in
// the sort).  The last partition writes small[kSmallTotal], and its clamp to the
// pair capacity with the overflow flag (device-sized chains: cap or dsz).
// Fused because at the sizes of one view it is launches that cost: the gather of the
// counts, a three-kernel scan and the clamp took 19 us of a 256 x 256 view's 220.
constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 8;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;

long long scan_scratch_words(long long n) { return 2 * ((n + SC_TILE - 1) / SC_TILE + 1); }

__global__ void __launch_bounds__(SC_THREADS) k_pair_offsets(const uint32_t *__restrict__ idx,
                                                             const uint32_t *__restrict__ count, long long n_all,
                                                             const uint32_t *__restrict__ d_all,
                                                             const uint32_t *__restrict__ d_n,
                                                             uint32_t *__restrict__ offs,
                                                             unsigned long long *__restrict__ status,
                                                             uint32_t *__restrict__ counter, uint32_t *__restrict__ small,
                                                             PairSlots slots, uint32_t cap,
                                                             const ChainSizes *__restrict__ dsz) {
    constexpr unsigned long long AGG = 1ull << 32, INC = 2ull << 32;
    __shared__ uint32_t s_warp[SC_THREADS / 32], s_part, s_excl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool fault = g_rs_fault == kFaultScan;  // (no kernel writes it: read ahead of the wait)
    const int limit = fault ? kFaultSpinLimit : kSpinLimit;
    chain_wait();
    if (d_all) n_all = *d_all;
    const long long n = d_n ? (long long)*d_n : n_all;
    const long long n_parts = (n + SC_TILE - 1) / SC_TILE;
    if (blockIdx.x >= n_parts) return;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_part = atomicAdd(counter, 1u);
        __syncthreads();
        const long long part = s_part;
        if (part >= n_parts) break;
        const long long base = part * SC_TILE + (long long)tid * SC_ITEMS;  // blocked per thread
        uint32_t v[SC_ITEMS], sum = 0;
#pragma unroll
        for (int i = 0; i < SC_ITEMS; ++i) {
            // (an entry outside the arrays, which only a sort that gave up can leave, has no pairs)
            const uint32_t k = base + i < n ? idx[base + i] : 0xFFFFFFFFu;
            v[i] = k < n_all ? count[k] : 0u;
            sum += v[i];
        }
        uint32_t x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        uint32_t before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < SC_THREADS / 32; ++w) {
            before += w < warp ? s_warp[w] : 0u;
            total += s_warp[w];
        }
        if (warp == 0) {
            volatile unsigned long long *st = status;
            if (lane == 0 && !(fault && part == 0)) atomicExch(status + part, (part == 0 ? INC : AGG) | total);
            uint32_t excl = 0;
            bool found = part == 0;
            for (long long p = part - 1; !found; p -= 32) {  // lane l: partition p - l
                unsigned long long s = p - lane >= 0 ? st[p - lane] : INC;
                for (int spins = 0; !(s & (AGG | INC)); ) {
                    if (++spins > limit) { atomicOr(small + slots.err, 1u); s = INC; break; }
                    __nanosleep(64);
                    s = st[p - lane];
                }
                __syncwarp();
                const unsigned inc = __ballot_sync(0xffffffffu, (s & INC) != 0);
                const int stop = inc ? __ffs(inc) - 1 : 31;  // nearest partition with its inclusive sum
                uint32_t c = lane <= stop ? (uint32_t)s : 0u;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
                excl += c;
                found = inc != 0;
            }
            if (lane == 0) {
                if (part > 0) atomicExch(status + part, INC | (unsigned long long)(excl + total));
                s_excl = excl;
            }
        }
        __syncthreads();
        uint32_t run = s_excl + before + x - sum;
#pragma unroll
        for (int i = 0; i < SC_ITEMS; ++i) {
            if (base + i < n) offs[base + i] = run;
            run += v[i];
        }
        if (part == n_parts - 1 && tid == SC_THREADS - 1) {
            if (dsz) cap = dsz->L_cap;
            small[slots.total] = run;
            small[slots.clamped] = run < cap ? run : cap;
            small[slots.overflow] = run > cap ? 1u : 0u;
        }
    }
}

void launch_pair_offsets(const uint32_t *idx, const uint32_t *count, long long n, const uint32_t *d_all,
                         const uint32_t *d_n, uint32_t *offs, uint32_t *scratch, uint32_t *counter, uint32_t *small,
                         const PairSlots &slots, uint32_t cap, const ChainSizes *dsz, cudaStream_t st) {
    if (n == 0) return;
    const long long parts = (n + SC_TILE - 1) / SC_TILE;
    const unsigned grid = (unsigned)std::min(parts, resident_ctas((const void *)k_pair_offsets, SC_THREADS));
    launch_chained(k_pair_offsets, grid, SC_THREADS, 0, st, idx, count, n, d_all, d_n, offs, (unsigned long long *)scratch,
                   counter, small, slots, cap, dsz);
}

}  // namespace dgs
