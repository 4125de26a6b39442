// Selecting the r largest scores of one unit by one CTA, candidates in registers: shared by the selection kernel and the
// kernel that copies the kept rows in the same launch.
#pragma once
#include <cuda_runtime.h>

#include "finch_internal.cuh"

namespace finch {
namespace pick {

constexpr int kMaxShort = 8192;  // candidates per unit: 1024 threads x 8
constexpr int kBins = 1024;
constexpr int kListed = 128;  // keys of one bin that are ranked directly

// Order-preserving key: larger score <=> larger key.  -0 is folded into +0; NaN gets key 0, below every number.
__device__ __forceinline__ uint32_t order_key(float s) {
    if (s != s) return 0u;
    uint32_t u = __float_as_uint(s);
    if ((u << 1) == 0u) u = 0u;  // -0 -> +0
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// What every unit starts with: its scores and output, how many to keep; false when there is nothing to do.  first: this
// CTA writes the request's length.
struct SelectUnit {
    const float *scores;
    int *kept;
    int N, r;
};
__device__ __forceinline__ bool select_unit(const ModelView &mv, const BatchView &bv, const UnitInfo &u, bool first,
                                            const float *scores, int *kept_idx, int *out_len, int *status, SelectUnit &s) {
    const int N = u.N;
    int r = bv.budget[u.b];
    r = r < N ? r : N;
    r = r < 0 ? 0 : r;
    if (!u.ok || r > u.cap || r > bv.max_budget) {  // block-uniform
        if (threadIdx.x == 0) {
            atomicOr(status, FINCH_DEV_BAD_BATCH);
            if (first) out_len[u.b] = 0;
        }
        return false;
    }
    if (first && threadIdx.x == 0) out_len[u.b] = r;
    s.scores = scores + ((int64_t)u.l * mv.G + u.G) * ((int64_t)bv.total_cache + bv.total_chunk) + u.cache0 + u.chunk0;
    s.kept = kept_idx + ((int64_t)u.l * mv.G + u.G) * bv.total_cache + u.cache0;
    s.N = N;
    s.r = r;
    return r > 0;
}

// The r largest of the unit's N scores, ties to the lower index; emit(rank, candidate) for each of them, ranks in index
// order.  All threads call it; N <= blockDim.x * kItems, blockDim.x a multiple of 32, 0 < r < N.
template <int kItems, typename Emit>
__device__ __forceinline__ void select_largest(const SelectUnit &s, const Emit &emit) {
    __shared__ __align__(16) int hist[kBins];
    __shared__ uint32_t warp_a[32], warp_b[32], listed[kListed];
    __shared__ int n_listed, sel_bin, sel_above, sel_count, sel_ties;
    __shared__ uint32_t sel_key;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;

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
        if (key[e] > T || (key[e] == T && eq < ties_to_keep)) emit(gt + min(eq, ties_to_keep), j0 + e);
        gt += key[e] > T;
        eq += key[e] == T;
    }
}

// Eight candidates per thread for long units (few barriers' worth of warps), four for short ones (latency).
inline int items_for(int max_n) { return max_n <= 2048 ? 4 : 8; }
inline int threads_for(int max_n) {
    const int items = items_for(max_n), threads = ((max_n + items - 1) / items + 31) / 32 * 32;
    return threads < 64 ? 64 : threads;
}

}  // namespace pick
}  // namespace finch
