// Top-r selection per (layer, selection group, request) without a sort, one CTA per unit.
//
// Scores are mapped to order-preserving 32-bit keys; the key T of the r-th largest score and the number of candidates
// strictly above it are found by counting, then an ordered sweep keeps every candidate above T plus the lowest-indexed
// candidates equal to T until r are kept, and writes the kept indices in increasing order.
//
//   select_kernel       units of at most 8192 candidates: keys in registers, a thread owns 4 or 8 consecutive candidates
//                       (select_core.cuh; a step of few units selects in the launch that copies the kept rows, compact.cu).
//                       The count runs over 1024 bins between the unit's smallest and largest key, so that scores of a
//                       narrow range still spread (8-bit digits of the whole key put most of them into one or two bins,
//                       whose atomics serialise); the few keys of the r-th one's bin are ranked directly.  Seven
//                       barriers in place of twenty.
//   select_long_kernel  longer units: four 8-bit radix passes over keys in shared memory, beyond 40960 in global memory.
#include "select_core.cuh"

namespace finch {
namespace {

using namespace pick;

constexpr int kLongThreads = 1024;
constexpr int kLongKeys = 40960;  // keys in shared memory

// a budget at or above the candidate count keeps everything, in order
__device__ __forceinline__ void keep_all(const SelectUnit &s) {
    for (int j = threadIdx.x; j < s.N; j += blockDim.x) s.kept[j] = j;
}

// The launcher gives N <= blockDim.x * kItems for every unit.
template <int kItems>
__global__ void __launch_bounds__(1024)
select_kernel(ModelView mv, BatchView bv, const float *scores, int *kept_idx, int *out_len, int *status) {
    dependency_wait();
    dependents_may_launch();
    SelectUnit s;
    if (!select_unit(mv, bv, unit_info(mv, bv, blockIdx.x, blockIdx.y), blockIdx.x == 0, scores, kept_idx, out_len, status, s)) return;
    if (s.r == s.N) return keep_all(s);
    select_largest<kItems>(s, [&](int rank, int j) { s.kept[rank] = j; });
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
    if (!select_unit(mv, bv, unit_info(mv, bv, blockIdx.x, blockIdx.y), blockIdx.x == 0, scores, kept_idx, out_len, status, s)) return;
    if (s.r == s.N) return keep_all(s);
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
        return launch_chained(items_for(max_n) == 4 ? select_kernel<4> : select_kernel<8>, grid, dim3(threads_for(max_n)), 0,
                              stream, mv, bv, scores, kept_idx, out_len, ctx.d_status);
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
