// Prompt-guided scoring with plain FMA dot products (fp32 inputs, head dimensions the tensor-core path does not take).
//
//   lse_simt     one CTA per (row tile of one query head, unit, key split): an online (max, sum-exp) per row over the
//                split's keys -> part (max of the base-2 logits, sum of exp2 against it)
//   colsum_simt  one CTA per (64 candidate keys, unit): merges the parts of each prompt row, then sweeps every prompt
//                row of every head of the group and accumulates exp2(s2 - max) / sum per key -> scores
//
// Keeping the row maximum and the reciprocal sum apart (instead of one log-sum-exp) keeps the exponent's argument
// a small difference even when the logits are large; both kernels form it with the same fused multiply-add
// (dot * scale2 - max), so the weight of a row's largest key is the same in the sum and in the column pass.
//
// A unit is one (layer, selection group, request).  Row tiles have 16, 32 or 64 rows, the least that holds the longest
// prompt; keys are split so that a small problem still fills the SMs (16 rows x 512 keys of 8 heads ran on 8 CTAs that
// walked the keys one tile after another: 57 us; 6 us over 64 CTAs).  A thread owns RM x 4 logits; both operands are staged
// as fp32 in slices of 32 dimensions, the next slice's loads in flight under the current one's arithmetic, and read as
// 128-bit vectors into packed multiply-adds.  All sums have a fixed order, so the scores are bit-identical from run to
// run.
#include "score_tc_common.cuh"

namespace finch {
namespace {

using tc::fma2;
using tc::unpack2;

constexpr int kKeys = 64;      // keys per CTA tile
constexpr int kSlice = 32;     // head_dim slice staged per iteration
constexpr int kPitch = kSlice + 4;  // floats per staged row: 128-bit reads of eight rows hit different banks
constexpr int kLanes = 16;     // key lanes: threads = row lanes (TY) x 16
constexpr int kMaxParts = 32;  // key splits

__device__ __forceinline__ float4 load4(const float *p) { return __ldg((const float4 *)p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
    const uint2 v = __ldg((const uint2 *)p);
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                       __uint_as_float(v.y & 0xffff0000u));
}

// A row-major operand tile of ROWS x d: where each of this thread's rows starts (null: no such row, zeros).
template <typename T, int ROWS, int THREADS>
struct Tile {
    static constexpr int kPer = ROWS * (kSlice / 4) / THREADS;  // float4 per thread and slice
    const T *row[kPer];
    float4 next[kPer];
    __device__ __forceinline__ static int row_of(int i) { return (threadIdx.x + i * THREADS) / (kSlice / 4); }
    __device__ __forceinline__ void fetch(int t0) {
        const int q = threadIdx.x % (kSlice / 4);
#pragma unroll
        for (int i = 0; i < kPer; ++i) next[i] = row[i] ? load4(row[i] + t0 + q * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void store(float *dst) const {
        const int q = threadIdx.x % (kSlice / 4);
#pragma unroll
        for (int i = 0; i < kPer; ++i) *(float4 *)(dst + row_of(i) * kPitch + q * 4) = next[i];
    }
};

template <typename T, int ROWS, int THREADS>
__device__ __forceinline__ void q_tile(Tile<T, ROWS, THREADS> &t, const TensorView &q, const UnitInfo &u, int h, int p0) {
    const T *base = (const T *)q.ptr + (int64_t)u.l * q.stride_layer + (int64_t)h * q.stride_head;
#pragma unroll
    for (int i = 0; i < Tile<T, ROWS, THREADS>::kPer; ++i) {
        const int p = p0 + t.row_of(i);
        t.row[i] = p < u.n_q ? base + (int64_t)(u.q0 + p) * q.stride_tok : nullptr;
    }
}
// candidate keys j0 .. of KV head kvh (cache rows first, then chunk rows)
template <typename T, int THREADS>
__device__ __forceinline__ void k_tile(Tile<T, kKeys, THREADS> &t, const TensorView &cache_k, const TensorView &chunk_k,
                                       const UnitInfo &u, int kvh, int j0) {
    const T *cbase = (const T *)cache_k.ptr + (int64_t)u.l * cache_k.stride_layer + (int64_t)kvh * cache_k.stride_head;
    const T *hbase = (const T *)chunk_k.ptr + (int64_t)u.l * chunk_k.stride_layer + (int64_t)kvh * chunk_k.stride_head;
#pragma unroll
    for (int i = 0; i < Tile<T, kKeys, THREADS>::kPer; ++i) {
        const int j = j0 + t.row_of(i);
        t.row[i] = j < u.c ? cbase + (int64_t)(u.cache0 + j) * cache_k.stride_tok
                           : (j < u.N ? hbase + (int64_t)(u.chunk0 + j - u.c) * chunk_k.stride_tok : nullptr);
    }
}

// acc[i][j] = Q[ty + TY i] . K[tx + 16 j] over all of head_dim; the even and the odd dimensions are summed apart.
template <typename T, int RM, int TY>
__device__ __forceinline__ void logits(float (&acc)[RM][4], Tile<T, RM * TY, TY * kLanes> &q, Tile<T, kKeys, TY * kLanes> &k, int d, float *qs, float *ks,
                                       int tx, int ty) {
    uint64_t sum[RM][4];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[i][j] = 0;
    q.fetch(0);
    k.fetch(0);
    for (int t0 = 0; t0 < d; t0 += kSlice) {
        __syncthreads();  // everyone is through with the previous slice
        q.store(qs);
        k.store(ks);
        __syncthreads();
        if (t0 + kSlice < d) {
            q.fetch(t0 + kSlice);
            k.fetch(t0 + kSlice);
        }
#pragma unroll 2
        for (int t = 0; t < kSlice; t += 4) {
            ulonglong2 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *(const ulonglong2 *)(ks + (tx + 16 * j) * kPitch + t);
#pragma unroll
            for (int i = 0; i < RM; ++i) {
                const ulonglong2 a = *(const ulonglong2 *)(qs + (ty + TY * i) * kPitch + t);
#pragma unroll
                for (int j = 0; j < 4; ++j) sum[i][j] = fma2(a.y, b[j].y, fma2(a.x, b[j].x, sum[i][j]));
            }
        }
    }
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float lo, hi;
            unpack2(sum[i][j], lo, hi);
            acc[i][j] = lo + hi;
        }
}

struct SimtParams {
    ModelView mv;
    BatchView bv;
    TensorView q, cache_k, chunk_k;
    float2 *parts;  // [splits][L][Hq][total_q] (max base-2 logit, sum of exp2 against it)
    float *row_lse, *scores;
    int splits;
    int head_ctas;  // CTAs a group's query heads are dealt to, each with scores of its own: 1, or one per head
    int early;  // the grid is resident at once: the next kernel may be scheduled
    int *status;
};

template <typename T, int RM, int TY>
__global__ void __launch_bounds__(TY * kLanes, 512 / (TY * kLanes))
lse_simt(SimtParams p) {
    __shared__ __align__(16) float qs[RM * TY * kPitch];
    __shared__ __align__(16) float ks[kKeys * kPitch];
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    dependency_wait();
    if (p.early) dependents_may_launch();
    const UnitInfo u = unit_info(mv, bv, blockIdx.y, blockIdx.z);
    if (!u.ok) {
        if (threadIdx.x == 0) atomicOr(p.status, FINCH_DEV_BAD_BATCH);
        return;
    }
    if (u.N == 0) return;
    constexpr int kRows = RM * TY;
    const int row_blocks = (bv.max_q + kRows - 1) / kRows;
    const int split = blockIdx.x % p.splits, rb = blockIdx.x / p.splits;
    const int hh = rb / row_blocks, p0 = (rb % row_blocks) * kRows;
    if (p0 >= u.n_q) return;
    const int h = u.G * mv.hpg + hh, kvh = h / mv.g;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const float scale2 = mv.scale * kLog2e;
    const int tiles = (u.N + kKeys - 1) / kKeys, per = (tiles + p.splits - 1) / p.splits;

    float run_max[RM], run_sum[RM];  // base-2 logits, over this thread's own key columns
    int vis[RM];                     // candidates the thread's rows attend to: all, or the row's limit (causal rows)
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        run_max[i] = -INFINITY;
        run_sum[i] = 0.f;
        const int pr = p0 + ty + TY * i;
        vis[i] = u.N;
        if (bv.row_limit && pr < u.n_q) vis[i] = max(0, min(u.N, bv.row_limit[u.q0 + pr]));
    }
    Tile<T, kRows, TY * kLanes> qt;
    Tile<T, kKeys, TY * kLanes> kt;
    q_tile(qt, p.q, u, h, p0);
    for (int t = split * per; t < min(tiles, (split + 1) * per); ++t) {
        const int j0 = t * kKeys;
        float acc[RM][4];
        k_tile(kt, p.cache_k, p.chunk_k, u, kvh, j0);
        logits<T, RM, TY>(acc, qt, kt, mv.d, qs, ks, tx, ty);
#pragma unroll
        for (int i = 0; i < RM; ++i) {
            float tile_max = -INFINITY;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + tx + 16 * j < vis[i]) tile_max = fmaxf(tile_max, acc[i][j] * scale2);
            if (tile_max == -INFINITY) continue;
            const float new_max = fmaxf(run_max[i], tile_max);
            float sum = run_sum[i] * exp2f(run_max[i] - new_max);  // exp2(-inf) = 0 on the first tile
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j0 + tx + 16 * j < vis[i]) sum += exp2f(fmaf(acc[i][j], scale2, -new_max));
            run_max[i] = new_max;
            run_sum[i] = sum;
        }
    }
    // merge the 16 column owners of each row (the lanes tx = 0..15 of a half warp) with a butterfly
    const int64_t rows_total = (int64_t)mv.L * mv.Hq * bv.total_q;
#pragma unroll
    for (int i = 0; i < RM; ++i) {
        float mx = run_max[i], sm = run_sum[i];
#pragma unroll
        for (int off = 1; off < 16; off <<= 1) {
            const float omx = __shfl_xor_sync(0xffffffffu, mx, off);
            const float osm = __shfl_xor_sync(0xffffffffu, sm, off);
            const float nmx = fmaxf(mx, omx);
            const float a = mx == -INFINITY ? 0.f : sm * exp2f(mx - nmx);
            const float b = omx == -INFINITY ? 0.f : osm * exp2f(omx - nmx);
            sm = a + b;  // commutative: both partners get the same bits
            mx = nmx;
        }
        const int pr = p0 + ty + TY * i;
        if (tx == 0 && pr < u.n_q)
            p.parts[split * rows_total + ((int64_t)u.l * mv.Hq + h) * bv.total_q + u.q0 + pr] = make_float2(mx, sm);
    }
}

// The parts of one row, merged in split order into (max, weight per unit of exp2): 1 / sum, times the fraction of the
// candidates the row sees when the per-row normalisation is on; a row that sees nothing weighs nothing.
__device__ __forceinline__ float2 merge_row_parts(const SimtParams &p, const UnitInfo &u, int64_t row, int vis, bool write_lse) {
    const int64_t rows_total = (int64_t)p.mv.L * p.mv.Hq * p.bv.total_q;
    float mx = -INFINITY, sm = 0.f;
    for (int i0 = 0; i0 < p.splits; i0 += 4) {
        float2 part[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            part[i] = i0 + i < p.splits ? p.parts[(i0 + i) * rows_total + row] : make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (part[i].y == 0.f) continue;  // a split that holds none of the row's keys (a NaN sum is the whole row's)
            const float nmx = fmaxf(mx, part[i].x);
            sm = sm * exp2f(mx - nmx) + part[i].y * exp2f(part[i].x - nmx);
            mx = nmx;
        }
    }
    if (p.bv.self_lse) {  // the keys the row attends to besides the candidates: one more term of the sum
        const float ex = p.bv.self_lse[row] * kLog2e;
        if (ex > -INFINITY) {
            const float nmx = fmaxf(mx, ex);
            sm = sm * exp2f(mx - nmx) + exp2f(ex - nmx);
            mx = nmx;
        }
    }
    if (write_lse) p.row_lse[row] = sm > 0.f ? (mx + log2f(sm)) * kLn2 : -INFINITY;
    float w = sm > 0.f ? 1.0f / sm : 0.f;
    if (p.bv.row_norm && p.bv.row_limit) w *= (float)vis / (float)u.N;
    return make_float2(sm > 0.f ? mx : 0.f, w);
}

template <typename T, int RM, int TY>
__global__ void __launch_bounds__(TY * kLanes, 512 / (TY * kLanes))
colsum_simt(SimtParams p) {
    constexpr int kRows = RM * TY;
    __shared__ __align__(16) float qs[kRows * kPitch];
    __shared__ __align__(16) float ks[kKeys * kPitch];
    __shared__ float2 stats[kRows];
    __shared__ int limits[kRows];
    __shared__ float red[TY][kKeys];
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    dependency_wait();
    if (p.early) dependents_may_launch();
    const UnitInfo u = unit_info(mv, bv, blockIdx.y / p.head_ctas, blockIdx.z);
    if (!u.ok) {
        if (threadIdx.x == 0) atomicOr(p.status, FINCH_DEV_BAD_BATCH);
        return;
    }
    const int h0 = p.head_ctas == 1 ? 0 : blockIdx.y % p.head_ctas, h1 = p.head_ctas == 1 ? mv.hpg : h0 + 1;
    const int j0 = blockIdx.x * kKeys;
    if (j0 >= u.N) return;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const float scale2 = mv.scale * kLog2e;

    float col[4] = {0.f, 0.f, 0.f, 0.f};
    Tile<T, kRows, TY * kLanes> qt;
    Tile<T, kKeys, TY * kLanes> kt;
    for (int hh = h0; hh < h1; ++hh) {
        const int h = u.G * mv.hpg + hh;
        k_tile(kt, p.cache_k, p.chunk_k, u, h / mv.g, j0);
        for (int p0 = 0; p0 < u.n_q; p0 += kRows) {
            __syncthreads();  // the previous row tile's statistics have been read
            if (threadIdx.x < kRows) {
                const int pr = p0 + threadIdx.x;
                float2 st = make_float2(0.f, 0.f);
                int lim = 0;  // keys at or beyond it are masked
                if (pr < u.n_q) {
                    lim = bv.row_limit ? max(0, min(u.N, bv.row_limit[u.q0 + pr])) : u.N;
                    st = merge_row_parts(p, u, ((int64_t)u.l * mv.Hq + h) * bv.total_q + u.q0 + pr, lim,
                                         p.row_lse && blockIdx.x == 0);
                }
                stats[threadIdx.x] = st;
                limits[threadIdx.x] = lim;
            }
            float acc[RM][4];
            q_tile(qt, p.q, u, h, p0);
            logits<T, RM, TY>(acc, qt, kt, mv.d, qs, ks, tx, ty);  // its barriers publish the statistics
#pragma unroll
            for (int i = 0; i < RM; ++i) {
                const float2 st = stats[ty + TY * i];
                const int lim = limits[ty + TY * i];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j0 + tx + 16 * j < lim) col[j] = fmaf(exp2f(fmaf(acc[i][j], scale2, -st.x)), st.y, col[j]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) red[ty][tx + 16 * j] = col[j];
    __syncthreads();
    if (threadIdx.x < kKeys && j0 + threadIdx.x < u.N) {
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < TY; ++r) s += red[r][threadIdx.x];
        p.scores[(int64_t)blockIdx.y * ((int64_t)bv.total_cache + bv.total_chunk) + u.cache0 + u.chunk0 + j0 + threadIdx.x] = s;
    }
}

template <typename T, int RM, int TY>
cudaError_t launch_t(const Ctx &ctx, SimtParams p, size_t capacity, cudaStream_t stream) {
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    const int units = mv.L * mv.G, sms = ctx.sm_count > 0 ? ctx.sm_count : 148;
    const int row_blocks = (bv.max_q + RM * TY - 1) / (RM * TY);
    const int key_tiles = (bv.max_cache + bv.max_chunk + kKeys - 1) / kKeys;
    if (units == 0 || bv.batch == 0 || row_blocks == 0 || key_tiles == 0) return cudaSuccess;
    // key splits: a wave of CTAs (an SM holds four of 128 threads, two of 256), at least one key tile each, as far as the scratch
    // goes.  Twice as many for the 256-thread tilings gain nothing (4 layers of 8 x 4 heads, 17 rows, 721 keys: 102.5 -> 98.8 us)
    constexpr int kResident = 512 / (TY * kLanes);
    const int64_t ctas = (int64_t)row_blocks * mv.hpg * units * bv.batch;
    const size_t rows = (size_t)mv.L * mv.Hq * (size_t)bv.total_q;
    int64_t splits = (kResident * (int64_t)sms + ctas - 1) / ctas;
    splits = min(splits, (int64_t)min(key_tiles, kMaxParts));
    if (rows) splits = min(splits, (int64_t)(capacity / rows));
    p.splits = splits < 1 ? 1 : (int)splits;
    p.early = ctas * p.splits <= kResident * sms;
    dim3 g1(row_blocks * mv.hpg * p.splits, units, bv.batch);
    cudaError_t e = launch_chained(lse_simt<T, RM, TY>, g1, dim3(TY * kLanes), 0, stream, p);
    if (e != cudaSuccess) return e;
    // Second sweep: with few key tiles the group's query heads go to CTAs of their own (their sums are added, in head
    // order, by one more small kernel) instead of being walked one after another (2 layers of 8 x 4 heads, 50 rows, 581
    // keys, fp32: the whole step 86 -> 76 us).
    const int64_t ctas2 = (int64_t)key_tiles * units * bv.batch;
    const size_t cand = (size_t)bv.total_cache + bv.total_chunk, head_scores = (size_t)units * mv.hpg * cand;
    float *const scores = p.scores;
    p.head_ctas = 1;
    if (mv.hpg > 1 && ctas2 < 2 * sms && units * mv.hpg <= 65535 && capacity >= rows * p.splits + (head_scores + 1) / 2) {
        p.head_ctas = mv.hpg;
        p.scores = (float *)(p.parts + rows * p.splits);
    }
    dim3 g2(key_tiles, units * p.head_ctas, bv.batch);
    p.early = ctas2 * p.head_ctas <= kResident * sms;
    ctx.launches += 2;
    e = launch_chained(colsum_simt<T, RM, TY>, g2, dim3(TY * kLanes), 0, stream, p);
    if (e != cudaSuccess || p.head_ctas == 1) return e;
    ModelView heads = mv;
    heads.G = mv.G * mv.hpg;
    return launch_sum_heads(ctx, heads, bv, p.scores, scores, mv.G, mv.hpg, stream);
}

template <typename T>
cudaError_t launch_rows(const Ctx &ctx, const SimtParams &p, size_t capacity, cudaStream_t stream) {
    if (p.bv.max_q <= 16) return launch_t<T, 2, 8>(ctx, p, capacity, stream);
    if (p.bv.max_q <= 32) return launch_t<T, 2, 16>(ctx, p, capacity, stream);
    return launch_t<T, 4, 16>(ctx, p, capacity, stream);
}

}  // namespace

cudaError_t launch_score_simt(const Ctx &ctx, const TensorView &q, const TensorView &cache_k, const TensorView &chunk_k,
                              const BatchView &bv, float *scores, float2 *scratch, size_t capacity, float *row_lse,
                              cudaStream_t stream) {
    SimtParams p{ctx.model, bv, q, cache_k, chunk_k, scratch, row_lse, scores, 1, 1, 0, ctx.d_status};
    return ctx.cfg.dtype == FINCH_F32 ? launch_rows<float>(ctx, p, capacity, stream)
                                      : launch_rows<__nv_bfloat16>(ctx, p, capacity, stream);
}

}  // namespace finch
