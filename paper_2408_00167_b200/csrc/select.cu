// Top-r selection per (layer, selection group, request) without a sort, one CTA per unit.
//
// Scores are mapped to order-preserving 32-bit keys; the key T of the r-th largest score and the number of candidates
// strictly above it are found by counting, then an ordered sweep keeps every candidate above T plus the lowest-indexed
// candidates equal to T until r are kept, and writes the kept indices in increasing order.
//
//   select_kernel       units of at most 8192 candidates: keys in registers, a thread owns 4 or 8 consecutive candidates.
//                       The count runs over 1024 bins between the unit's smallest and largest key, so that scores of a
//                       narrow range still spread (8-bit digits of the whole key put most of them into one or two bins,
//                       whose atomics serialise); the few keys of the r-th one's bin are ranked directly.  Seven
//                       barriers in place of twenty.
//   select_long_kernel  longer units: four 8-bit radix passes over keys in shared memory, beyond 40960 in global memory.
#include "finch_internal.cuh"

namespace finch {
namespace {

constexpr int kLongThreads = 1024;
constexpr int kLongKeys = 40960;  // keys in shared memory
constexpr int kMaxShort = 8192;  // candidates per unit of select_kernel: 1024 threads x 8
constexpr int kBins = 1024;
constexpr int kListed = 128;  // keys of one bin that are ranked directly

// Order-preserving key: larger score <=> larger key.  -0 is folded into +0; NaN gets key 0, below every number.
__device__ __forceinline__ uint32_t order_key(float s) {
    if (s != s) return 0u;
    uint32_t u = __float_as_uint(s);
    if ((u << 1) == 0u) u = 0u;  // -0 -> +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// What every unit starts with: its scores and output, how many to keep; false when there is nothing (more) to do.
struct SelectUnit {
    const float *scores;
    int *kept;
    int N, r;
};
__device__ __forceinline__ bool select_unit(const ModelView &mv, const BatchView &bv, const float *scores, int *kept_idx,
                                            int *out_len, int *status, SelectUnit &s) {
    const int unit = blockIdx.x;
    const UnitInfo u = unit_info(mv, bv, unit, blockIdx.y);
    const int N = u.N;
    int r = bv.budget[u.b];
    r = r < N ? r : N;
    r = r < 0 ? 0 : r;
    if (!u.ok || r > u.cap || r > bv.max_budget) {  // block-uniform
        if (threadIdx.x == 0) {
            atomicOr(status, FINCH_DEV_BAD_BATCH);
            if (unit == 0) out_len[u.b] = 0;
        }
        return false;
    }
    if (unit == 0 && threadIdx.x == 0) out_len[u.b] = r;
    s.scores = scores + ((int64_t)u.l * mv.G + u.G) * ((int64_t)bv.total_cache + bv.total_chunk) + u.cache0 + u.chunk0;
    s.kept = kept_idx + ((int64_t)u.l * mv.G + u.G) * bv.total_cache + u.cache0;
    s.N = N;
    s.r = r;
    if (r == N)  // a budget at or above the candidate count keeps everything, in order
        for (int j = threadIdx.x; j < N; j += blockDim.x) s.kept[j] = j;
    return r > 0 && r < N;
}

// The launcher gives N <= blockDim.x * kItems for every unit.
template <int kItems>
__global__ void __launch_bounds__(1024)
select_kernel(ModelView mv, BatchView bv, const float *scores, int *kept_idx, int *out_len, int *status) {
    __shared__ __align__(16) int hist[kBins];
    __shared__ uint32_t warp_a[32], warp_b[32], listed[kListed];
    __shared__ int n_listed, sel_bin, sel_above, sel_count, sel_ties;
    __shared__ uint32_t sel_key;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;

    dependency_wait();
    dependents_may_launch();
    SelectUnit s;
    if (!select_unit(mv, bv, scores, kept_idx, out_len, status, s)) return;

    const int j0 = threadIdx.x * kItems, mine = max(0, min(kItems, s.N - j0));  // this thread's candidates
    uint32_t key[kItems], lo = 0xffffffffu, hi = 0;
#pragma unroll
    for (int e = 0; e < kItems; ++e) key[e] = e < mine ? __float_as_uint(s.scores[j0 + e]) : 0u;
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
        key[e] = order_key(__uint_as_float(key[e]));
        if (e < mine) {
            lo = min(lo, key[e]);
            hi = max(hi, key[e]);
        }
    }
    for (int i = threadIdx.x; i < kBins; i += blockDim.x) hist[i] = 0;
    if (threadIdx.x == 0) n_listed = 0;
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        warp_a[warp] = lo;
        warp_b[warp] = hi;
    }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lane < n_warps ? warp_a[lane] : 0xffffffffu);
    hi = __reduce_max_sync(0xffffffffu, lane < n_warps ? warp_b[lane] : 0u);

    // ---- the remaining-th largest of the keys in [lo, hi]; every round shrinks the range a thousandfold
    int remaining = s.r;
    uint32_t T;
    for (;;) {
        const uint32_t range = hi - lo;
        const int shift = max(0, 22 - __clz(range));  // range >> shift < 1024
#pragma unroll
        for (int e = 0; e < kItems; ++e)
            if (e < mine && key[e] - lo <= range) atomicAdd(&hist[(key[e] - lo) >> shift], 1);
        __syncthreads();
        // thread i owns a run of bins, the largest keys first; find the bin in which the running count reaches `remaining`
        const int per = (kBins + blockDim.x - 1) / blockDim.x, top = kBins - 1 - threadIdx.x * per;
        int count = 0;
        for (int i = 0; i < per; ++i)
            if (top - i >= 0) count += hist[top - i];
        int incl = count;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += v;
        }
        if (lane == 31) warp_a[warp] = incl;
        __syncthreads();
        const uint32_t before = lane < warp ? warp_a[lane] : 0u;
        int above = (int)__reduce_add_sync(0xffffffffu, before) + incl - count;
        if (above < remaining && remaining <= above + count) {
            for (int i = 0; i < per; ++i) {
                const int c = hist[top - i];
                if (remaining <= above + c) {
                    sel_bin = top - i;
                    sel_above = above;
                    sel_count = c;
                    break;
                }
                above += c;
            }
        }
        __syncthreads();
        remaining -= sel_above;
        lo += (uint32_t)sel_bin << shift;
        hi = lo + min(hi - lo, (1u << shift) - 1u);
        T = lo;
        if (shift == 0) break;  // a bin is a single key
        if (sel_count <= kListed) {
#pragma unroll
            for (int e = 0; e < kItems; ++e)
                if (e < mine && key[e] - lo <= hi - lo) listed[atomicAdd(&n_listed, 1)] = key[e];
            __syncthreads();
            for (int i = threadIdx.x; i < sel_count; i += blockDim.x) {
                const uint32_t k = listed[i];
                int gt = 0, ge = 0;
                for (int q = 0; q < sel_count; ++q) {
                    gt += listed[q] > k;
                    ge += listed[q] >= k;
                }
                if (gt < remaining && remaining <= ge) {  // equal keys write the same values
                    sel_key = k;
                    sel_ties = remaining - gt;
                }
            }
            __syncthreads();
            T = sel_key;
            remaining = sel_ties;
            break;
        }
        for (int i = threadIdx.x; i < kBins; i += blockDim.x) hist[i] = 0;
        __syncthreads();
    }
    const int ties_to_keep = remaining;  // >= 1

    // ---- ordered sweep: keep key > T, and the first `ties_to_keep` keys == T.  One block-wide scan of (above, equal).
    uint32_t n = 0;
#pragma unroll
    for (int e = 0; e < kItems; ++e)
        if (e < mine) n += key[e] > T ? 0x10000u : (key[e] == T ? 1u : 0u);
    uint32_t incl = n;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) warp_b[warp] = incl;
    __syncthreads();
    const uint32_t at = __reduce_add_sync(0xffffffffu, lane < warp ? warp_b[lane] : 0u) + incl - n;
    int gt = at >> 16, eq = at & 0xffffu;
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
        if (e >= mine) continue;
        if (key[e] > T || (key[e] == T && eq < ties_to_keep)) s.kept[gt + min(eq, ties_to_keep)] = j0 + e;
        gt += key[e] > T;
        eq += key[e] == T;
    }
}

// 32 registers per thread: two CTAs of 1024 threads per SM
__global__ void __launch_bounds__(kLongThreads, 2)
select_long_kernel(ModelView mv, BatchView bv, const float *scores, int *kept_idx, int *out_len, int smem_keys, int *status) {
    constexpr int kSelThreads = kLongThreads;
    constexpr int kSelWarps = kSelThreads / 32;
    extern __shared__ uint32_t key_cache[];  // the first min(N, smem_keys) keys
    __shared__ int hist[256];
    __shared__ int warp_tot[2][kSelWarps];
    __shared__ int sel_digit, sel_above;

    dependency_wait();
    dependents_may_launch();
    SelectUnit s;
    if (!select_unit(mv, bv, scores, kept_idx, out_len, status, s)) return;
    const float *sc = s.scores;
    int *kept = s.kept;
    const int N = s.N, r = s.r;

    const int n_cached = N < smem_keys ? N : smem_keys;
    for (int j = threadIdx.x; j < n_cached; j += kSelThreads) key_cache[j] = order_key(sc[j]);
    __syncthreads();
    auto key_at = [&](int j) -> uint32_t { return j < n_cached ? key_cache[j] : order_key(sc[j]); };

    // ---- radix search for the r-th largest key
    uint32_t prefix = 0, mask = 0;
    int remaining = r;  // rank, among the keys matching the prefix, of the key we look for (1 = largest)
    for (int shift = 24; shift >= 0; shift -= 8) {
        if (threadIdx.x < 256) hist[threadIdx.x] = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < N; j += kSelThreads) {
            const uint32_t k = key_at(j);
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // lane i owns digits 255-8i .. 248-8i (descending); find the digit where the running count reaches
            // `remaining`
            const int lane = threadIdx.x;
            int mine = 0;
#pragma unroll
            for (int t = 0; t < 8; ++t) mine += hist[255 - 8 * lane - t];
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            int above = incl - mine;
            if (above < remaining && remaining <= incl) {
                for (int t = 0; t < 8; ++t) {
                    const int digit = 255 - 8 * lane - t;
                    const int cnt = hist[digit];
                    if (remaining <= above + cnt) {
                        sel_digit = digit;
                        sel_above = above;
                        break;
                    }
                    above += cnt;
                }
            }
        }
        __syncthreads();
        prefix |= (uint32_t)sel_digit << shift;
        mask |= 255u << shift;
        remaining -= sel_above;
        __syncthreads();
    }
    const uint32_t T = prefix;
    const int ties_to_keep = remaining;  // >= 1

    // ---- ordered sweep: keep key > T, and the first `ties_to_keep` keys == T.  A thread takes four consecutive
    // candidates, so two block-wide exclusive scans per 4096 candidates (ties before me, kept before me) place every
    // kept index; the output is ascending by construction.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto block_scan = [&](int v, int *buf, int &total) -> int {  // exclusive prefix of v over the block, in thread order
        int incl = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += up;
        }
        if (lane == 31) buf[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            int t = lane < kSelWarps ? buf[lane] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, t, off);
                if (lane >= off) t += up;
            }
            if (lane < kSelWarps) buf[lane] = t;  // inclusive totals of the warps
        }
        __syncthreads();
        total = buf[kSelWarps - 1];
        return (warp ? buf[warp - 1] : 0) + incl - v;
    };
    constexpr int kPerThread = 4;
    int base_eq = 0, base_keep = 0;
    for (int j0 = 0; j0 < N; j0 += kSelThreads * kPerThread) {
        const int j = j0 + threadIdx.x * kPerThread;
        uint32_t k[kPerThread];
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) k[e] = j + e < N ? key_at(j + e) : 0u;
        int n_eq = 0;
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) n_eq += (j + e < N && k[e] == T) ? 1 : 0;
        int eq_all;
        int eq_before = base_eq + block_scan(n_eq, warp_tot[0], eq_all);
        bool keep[kPerThread];
        int n_keep = 0;
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            const bool in = j + e < N;
            const bool eq = in && k[e] == T;
            keep[e] = in && (k[e] > T || (eq && eq_before < ties_to_keep));
            eq_before += eq ? 1 : 0;
            n_keep += keep[e] ? 1 : 0;
        }
        int keep_all;
        int slot = base_keep + block_scan(n_keep, warp_tot[1], keep_all);
#pragma unroll
        for (int e = 0; e < kPerThread; ++e)
            if (keep[e]) kept[slot++] = j + e;
        base_eq += eq_all;
        base_keep += keep_all;
        // the next iteration's first scan writes warp_tot[0] after this iteration's last barrier, and warp_tot[1]
        // after two more: every read above has been made by then
    }
}

}  // namespace

cudaError_t launch_select(const Ctx &ctx, const float *scores, const BatchView &bv, int *kept_idx, int *out_len,
                          cudaStream_t stream) {
    const ModelView &mv = ctx.model;
    const int units = mv.L * mv.G;
    if (units == 0 || bv.batch == 0) return cudaSuccess;
    const int max_n = bv.max_cache + bv.max_chunk;
    dim3 grid(units, bv.batch);
    ctx.launches += 1;
    if (max_n <= kMaxShort) {
        // eight candidates per thread for long units (few barriers' worth of warps), four for short ones (latency)
        const int items = max_n <= 2048 ? 4 : 8;
        const int threads = max(64, ((max_n + items - 1) / items + 31) / 32 * 32);
        return launch_chained(items == 4 ? select_kernel<4> : select_kernel<8>, grid, dim3(threads), 0, stream, mv, bv, scores,
                              kept_idx, out_len, ctx.d_status);
    }
    const int smem_keys = max_n < kLongKeys ? max_n : kLongKeys;  // up to 160 KiB on chip; longer inputs re-read global
    if (!ctx.smem_ready(kSmemSelect)) {
        cudaError_t e = cudaFuncSetAttribute(select_long_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLongKeys * 4);
        if (e != cudaSuccess) return e;
        ctx.smem_set(kSmemSelect);
    }
    return launch_chained(select_long_kernel, grid, dim3(kLongThreads), (size_t)smem_keys * sizeof(uint32_t), stream, mv, bv,
                          scores, kept_idx, out_len, smem_keys, ctx.d_status);
}

}  // namespace finch
