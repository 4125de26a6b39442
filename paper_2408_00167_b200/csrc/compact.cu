// Cache compaction: gather the kept K/V rows and positions into the next cache, in kept (ascending) order.
//
// One CTA copies a block of output rows of one KV head of one request, K and V, as 16-byte pieces: consecutive threads
// move consecutive pieces of a row, so both the gathered reads (whole rows) and the writes (contiguous rows) are fully
// coalesced 128-bit accesses, and every thread has eight loads in flight before its first store.  The dependent chain
// in front of the copies (batch metadata -> kept indices -> source addresses) wants large blocks, 256 rows where they
// fill the chip twice over (c. 92 % of the copy rate); smaller problems take smaller blocks so that every SM has some.
// KV heads are spread over the grid also where one selection group covers them all (32 heads in a CTA's loop left a
// 32-layer step with 128 CTAs: 0.49 ms for 1 GB, re-positioned).
#include <cuda_bf16.h>

#include <type_traits>

#include "select_core.cuh"

namespace finch {
namespace {

constexpr int kCompactThreads = 256;
constexpr int kMaxRowsPerCta = kCompactThreads;  // one thread fetches one kept index
constexpr int kMinRowsPerCta = 16;

// ---- rotary re-positioning (Method, "Managing the Cache"): a kept key that moves from candidate index j to output
// slot i is rotated by delta = i - j positions; pair t of the row turns by delta * theta^(-2t/d).  Cosine and sine
// come from the context's table (computed in double, one row per distance |delta|; a negative delta flips the sine's
// sign), the rotation itself is fp32, the result is rounded to the storage type.
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {  // both rounded to nearest even, one instruction
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *(const uint32_t *)&v;
}
__device__ __forceinline__ void rotate_pair(float x, float y, float2 cs, float sign, float &xo, float &yo) {
    const float sn = cs.y * sign;
    xo = fmaf(x, cs.x, -(y * sn));
    yo = fmaf(y, cs.x, x * sn);
}
// 16 bytes of x coordinates and the 16 bytes of their partners (kElems pairs, pairs (t, t + d/2)), rotated in place.
// cs points at the table entries of the kElems pairs.
template <int kElems>
__device__ __forceinline__ void rotate_pieces(uint4 &px, uint4 &py, const float2 *cs, float sign) {
    uint32_t *wx = (uint32_t *)&px, *wy = (uint32_t *)&py;
    float2 t[kElems];
#pragma unroll
    for (int e = 0; e < kElems / 2; ++e) {
        const float4 two = __ldg((const float4 *)cs + e);
        t[2 * e] = make_float2(two.x, two.y);
        t[2 * e + 1] = make_float2(two.z, two.w);
    }
    if (kElems == 4) {  // fp32
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float xo, yo;
            rotate_pair(__uint_as_float(wx[e]), __uint_as_float(wy[e]), t[e], sign, xo, yo);
            wx[e] = __float_as_uint(xo);
            wy[e] = __float_as_uint(yo);
        }
    } else {  // bf16, two per word
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float x0, y0, x1, y1;
            rotate_pair(bf16_lo(wx[e]), bf16_lo(wy[e]), t[2 * e], sign, x0, y0);
            rotate_pair(bf16_hi(wx[e]), bf16_hi(wy[e]), t[2 * e + 1], sign, x1, y1);
            wx[e] = pack_bf16(x0, x1);
            wy[e] = pack_bf16(y0, y1);
        }
    }
}
// One 16-byte piece whose pairs are neighbouring coordinates (2t, 2t + 1): kElems / 2 pairs.
template <int kElems>
__device__ __forceinline__ void rotate_interleaved(uint4 &pv, const float2 *cs, float sign) {
    uint32_t *w = (uint32_t *)&pv;
    float2 t[kElems / 2];
#pragma unroll
    for (int e = 0; e < kElems / 4; ++e) {
        const float4 two = __ldg((const float4 *)cs + e);
        t[2 * e] = make_float2(two.x, two.y);
        t[2 * e + 1] = make_float2(two.z, two.w);
    }
    if (kElems == 4) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float xo, yo;
            rotate_pair(__uint_as_float(w[2 * e]), __uint_as_float(w[2 * e + 1]), t[e], sign, xo, yo);
            w[2 * e] = __float_as_uint(xo);
            w[2 * e + 1] = __float_as_uint(yo);
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float xo, yo;
            rotate_pair(bf16_lo(w[e]), bf16_hi(w[e]), t[e], sign, xo, yo);
            w[e] = pack_bf16(xo, yo);
        }
    }
}

// Rows of one tensor (K or V of a KV head): where candidate j's row starts, and output row i.
struct RowMap {
    const char *cache, *chunk;
    char *out;
    int64_t cache_step, chunk_step, out_step;
    int c;
    __device__ RowMap(const UnitInfo &u, int kvh, int i0, int64_t e, const TensorView &ca, const TensorView &ch,
                      const TensorView &dst) {
        cache = ca.ptr + ((int64_t)u.l * ca.stride_layer + (int64_t)kvh * ca.stride_head + (int64_t)u.cache0 * ca.stride_tok) * e;
        chunk = ch.ptr + ((int64_t)u.l * ch.stride_layer + (int64_t)kvh * ch.stride_head +
                          (int64_t)(u.chunk0 - u.c) * ch.stride_tok) * e;
        out = const_cast<char *>(dst.ptr) + ((int64_t)u.l * dst.stride_layer + (int64_t)kvh * dst.stride_head +
                                             (int64_t)(u.cache0 + i0) * dst.stride_tok) * e;
        cache_step = ca.stride_tok * e;
        chunk_step = ch.stride_tok * e;
        out_step = dst.stride_tok * e;
        c = u.c;
    }
    __device__ const char *src(int j) const { return j < c ? cache + j * cache_step : chunk + j * chunk_step; }
};

// Plain copies.  A thread keeps its piece of the row and walks the rows threads / pieces apart.
__device__ __forceinline__ void copy_rows(const RowMap &m, const int *src_idx, int rows, int pieces, int threads) {
    constexpr int kBatch = 8;
    const int step = threads / pieces, r0 = threadIdx.x / pieces, off = (threadIdx.x - r0 * pieces) * 16;
    if (r0 >= step) return;
#pragma unroll 1
    for (int r = r0; r < rows; r += step * kBatch) {
        uint4 v[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {  // all of this batch's loads first ..
            const int row = r + k * step, j = row < rows ? src_idx[row] : -1;
            if (j >= 0) v[k] = __ldcs((const uint4 *)(m.src(j) + off));
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {  // .. then its stores
            const int row = r + k * step;
            if (row < rows && src_idx[row] >= 0) *(uint4 *)(m.out + row * m.out_step + off) = v[k];
        }
    }
}

// Copies with rotation, four rows in flight.  kSplit: pairs (t, t + d/2), a thread moves a piece of the row's first half
// and the partner piece of the second; else pairs (2t, 2t + 1) inside a piece.
template <int kElems, bool kSplit>
__device__ __forceinline__ void rotate_rows(const RowMap &m, const int *src_idx, int rows, int i0, int d, int elem_bytes,
                                            const float2 *rope_table, int threads) {
    constexpr int kBatch = 4;
    const int half = d / 2, pieces = d * elem_bytes / 16 / (kSplit ? 2 : 1);
    const int step = threads / pieces, r0 = threadIdx.x / pieces, piece = threadIdx.x - r0 * pieces;
    const int off = piece * 16, far = half * elem_bytes;
    const float2 *table = rope_table + piece * (kSplit ? kElems : kElems / 2);
    if (r0 >= step) return;
#pragma unroll 1
    for (int r = r0; r < rows; r += step * kBatch) {
        uint4 a[kBatch], b[kSplit ? kBatch : 1];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int row = r + k * step, j = row < rows ? src_idx[row] : -1;
            if (j >= 0) {
                const char *src = m.src(j) + off;
                a[k] = __ldcs((const uint4 *)src);
                if (kSplit) b[k] = __ldcs((const uint4 *)(src + far));
            }
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int row = r + k * step, j = row < rows ? src_idx[row] : -1;
            if (j < 0) continue;
            const int delta = i0 + row - j;
            const float2 *cs = table + (int64_t)abs(delta) * half;
            const float sign = delta < 0 ? -1.f : 1.f;
            char *dst = m.out + row * m.out_step + off;
            if (kSplit) {
                rotate_pieces<kElems>(a[k], b[k], cs, sign);
                *(uint4 *)(dst + far) = b[k];
            } else {
                rotate_interleaved<kElems>(a[k], cs, sign);
            }
            *(uint4 *)dst = a[k];
        }
    }
}

struct CompactTensors {
    TensorView cache_k, cache_v, chunk_k, chunk_v, out_k, out_v;
    const int *cache_pos, *chunk_pos;
    int *out_pos;
};

// Source of output row i of a group: checks the index, and writes the row's position where `leader` (the CTA of the
// group's first KV head).  -1: no copy.
template <int ROPE>
__device__ __forceinline__ int place_row(const ModelView &mv, const UnitInfo &u, const CompactTensors &t, int64_t unit_off,
                                         bool leader, int i, int j, int *status) {
    // with rotation a distance beyond the table (only possible when out_len exceeds the candidate count) is refused
    if (j < 0 || j >= u.N || (ROPE && abs(i - j) >= mv.rope_rows)) {
        atomicOr(status, FINCH_DEV_BAD_INDEX);
        return -1;
    }
    if (leader) t.out_pos[unit_off + i] = j < u.c ? t.cache_pos[unit_off + j] : t.chunk_pos[u.chunk0 + j - u.c];
    return j;
}

// ROPE 0: bit-for-bit copies; 1 / 2: K rows re-positioned, pairs (t, t + d/2) / (2t, 2t + 1).
template <int ROPE, int kElems>
__device__ __forceinline__ void move_rows(const ModelView &mv, const UnitInfo &u, int kvh, int i0, int rows,
                                          const int *src_idx, const CompactTensors &t, int threads) {
    const int pieces = mv.d * mv.elem_bytes / 16;  // 16-byte pieces per row
    const RowMap k_rows(u, kvh, i0, mv.elem_bytes, t.cache_k, t.chunk_k, t.out_k);
    if (ROPE)
        rotate_rows<kElems, ROPE == 1>(k_rows, src_idx, rows, i0, mv.d, mv.elem_bytes, mv.rope_table, threads);
    else
        copy_rows(k_rows, src_idx, rows, pieces, threads);
    copy_rows(RowMap(u, kvh, i0, mv.elem_bytes, t.cache_v, t.chunk_v, t.out_v), src_idx, rows, pieces, threads);
}

template <int ROPE, int kElems>
__global__ void __launch_bounds__(kCompactThreads)
compact_kernel(ModelView mv, BatchView bv, const int *kept_idx, const int *out_len, CompactTensors t, int rows_per_cta, int *status) {
    __shared__ int src_idx[kMaxRowsPerCta];
    dependency_wait();  // no early launch of the next kernel: this grid runs in many waves and needs every slot
    const int l = blockIdx.y / mv.Hkv, kvh = blockIdx.y - l * mv.Hkv, group = kvh / mv.kvpg;
    const UnitInfo u = unit_info(mv, bv, l * mv.G + group, blockIdx.z);
    if (!u.ok) {
        if (threadIdx.x == 0) atomicOr(status, FINCH_DEV_BAD_BATCH);
        return;
    }
    int r = out_len[u.b];
    if (r > u.cap) r = u.cap;
    const int i0 = blockIdx.x * rows_per_cta;
    if (i0 >= r) return;
    const int rows = min(rows_per_cta, r - i0);
    const int64_t unit_off = ((int64_t)u.l * mv.G + u.G) * bv.total_cache + u.cache0;
    if (threadIdx.x < rows)
        src_idx[threadIdx.x] = place_row<ROPE>(mv, u, t, unit_off, kvh == group * mv.kvpg, i0 + threadIdx.x,
                                               kept_idx[unit_off + i0 + threadIdx.x], status);
    __syncthreads();
    move_rows<ROPE, kElems>(mv, u, kvh, i0, rows, src_idx, t, kCompactThreads);
}

// Selection and copies in one launch, for steps whose copies are a single wave of CTAs: every CTA selects for its unit
// (the scores come from L2) and copies its own block of the kept rows, so the kept indices need not travel through
// global memory and a launch to reach the copies.  Bound by latency: one layer of 8 KV heads, whole step, 4096 candidates
// 39.3 -> 35.2 us, 1024 candidates 24.0 -> 21.7, 512 candidates in fp32 17.4 -> 16.0; 9 layers of 944: 50.3 -> 46.5.
constexpr int kPickThreads = 512, kMaxRowsPicked = 512;
template <int ROPE, int kElems, int kItems>
__global__ void __launch_bounds__(kPickThreads)
select_compact_kernel(ModelView mv, BatchView bv, const float *scores, int *kept_idx, int *out_len, CompactTensors t,
                      int rows_per_cta, int *status) {
    __shared__ int src_idx[kMaxRowsPicked];
    dependency_wait();
    dependents_may_launch();  // the whole grid is resident (see launch_select_compact)
    const int l = blockIdx.y / mv.Hkv, kvh = blockIdx.y - l * mv.Hkv, group = kvh / mv.kvpg;
    const UnitInfo u = unit_info(mv, bv, l * mv.G + group, blockIdx.z);
    const bool leader = kvh == group * mv.kvpg;
    pick::SelectUnit s;
    if (!pick::select_unit(mv, bv, u, blockIdx.x == 0 && blockIdx.y == 0, scores, kept_idx, out_len, status, s)) return;
    const int i0 = blockIdx.x * rows_per_cta, rows = min(rows_per_cta, s.r - i0);
    if (rows <= 0) return;
    if (s.r == s.N) {  // everything, in order
        for (int i = threadIdx.x; i < rows; i += blockDim.x) src_idx[i] = i0 + i;
    } else {
        pick::select_largest<kItems>(s, [&](int rank, int j) {
            if ((unsigned)(rank - i0) < (unsigned)rows) src_idx[rank - i0] = j;
        });
    }
    __syncthreads();
    const int64_t unit_off = ((int64_t)u.l * mv.G + u.G) * bv.total_cache + u.cache0;
    if (leader || ROPE) {
        for (int i = threadIdx.x; i < rows; i += blockDim.x) {
            const int j = src_idx[i], from = place_row<ROPE>(mv, u, t, unit_off, leader, i0 + i, j, status);
            if (leader) s.kept[i0 + i] = j;
            if (ROPE) src_idx[i] = from;
        }
    }
    if (ROPE) __syncthreads();
    move_rows<ROPE, kElems>(mv, u, kvh, i0, rows, src_idx, t, blockDim.x);
}

// The kernel of a rotation mode: f(mode, elements per 16 bytes).
template <typename F>
auto by_rotation(const ModelView &mv, const F &f) {
    const bool f32 = mv.elem_bytes == 4;
    using Std = std::integral_constant<int, 1>;
    if (!(mv.rope_theta > 0.f)) return f(std::integral_constant<int, 0>(), std::integral_constant<int, 8>());
    if (mv.rope_pairing == 0)
        return f32 ? f(Std(), std::integral_constant<int, 4>()) : f(Std(), std::integral_constant<int, 8>());
    return f32 ? f(std::integral_constant<int, 2>(), std::integral_constant<int, 4>())
               : f(std::integral_constant<int, 2>(), std::integral_constant<int, 8>());
}

// CTAs of kCompactThreads of the selecting kernel that an SM holds at a time.
int picks_per_sm(const Ctx &ctx, const ModelView &mv, int items) {
    return by_rotation(mv, [&](auto rope, auto elems) -> int {
        constexpr int kRope = decltype(rope)::value, kElems = decltype(elems)::value;
        int8_t &known = ctx.picks[kRope][kElems == 8][items == 4];
        if (known) return known;
        int n = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &n, items == 4 ? select_compact_kernel<kRope, kElems, 4> : select_compact_kernel<kRope, kElems, 8>, kCompactThreads,
                0) != cudaSuccess) {
            (void)cudaGetLastError();
            return 1;
        }
        n = n > 3 ? 3 : n;  // measured with three
        if (ctx.on_own_device()) known = (int8_t)n;
        return n;
    });
}

}  // namespace

cudaError_t launch_compact(const Ctx &ctx, const int *kept_idx, const int *out_len, const TensorView &cache_k,
                           const TensorView &cache_v, const int *cache_pos, const TensorView &chunk_k,
                           const TensorView &chunk_v, const int *chunk_pos, const BatchView &bv, const TensorView &out_k,
                           const TensorView &out_v, int *out_pos, cudaStream_t stream) {
    const ModelView &mv = ctx.model;
    const int heads = mv.L * mv.Hkv;
    if (heads == 0 || bv.batch == 0 || bv.max_budget == 0) return cudaSuccess;
    // the largest block that still gives every SM two CTAs
    const int64_t sms = ctx.sm_count > 0 ? ctx.sm_count : 148;
    int rows = kMaxRowsPerCta;
    while (rows > kMinRowsPerCta && (int64_t)((bv.max_budget + rows - 1) / rows) * heads * bv.batch < 2 * sms) rows /= 2;
    dim3 grid((bv.max_budget + rows - 1) / rows, heads, bv.batch);
    ctx.launches += 1;
    const CompactTensors t{cache_k, cache_v, chunk_k, chunk_v, out_k, out_v, cache_pos, chunk_pos, out_pos};
    return by_rotation(mv, [&](auto rope, auto elems) {
        return launch_chained(compact_kernel<decltype(rope)::value, decltype(elems)::value>, grid, dim3(kCompactThreads), 0, stream,
                              mv, bv, kept_idx, out_len, t, rows, ctx.d_status);
    });
}

cudaError_t launch_select_compact(const Ctx &ctx, const float *scores, const TensorView &cache_k, const TensorView &cache_v,
                                  const int *cache_pos, const TensorView &chunk_k, const TensorView &chunk_v,
                                  const int *chunk_pos, const BatchView &bv, const TensorView &out_k, const TensorView &out_v,
                                  int *out_pos, int *kept_idx, int *out_len, cudaStream_t stream) {
    const ModelView &mv = ctx.model;
    const int max_n = bv.max_cache + bv.max_chunk, heads = mv.L * mv.Hkv;
    const int64_t sms = ctx.sm_count > 0 ? ctx.sm_count : 148, units = (int64_t)heads * bv.batch;
    // Threads for the copies even where the selection needs fewer (96 threads: 57 us for a step of 43).  A unit's rows are
    // cut evenly into as many blocks as give every SM a CTA, two of short units (two CTAs of 512 threads per SM select
    // twice as often for blocks of half the rows: 42 us against 35); at most a wave, as many CTAs of 256 threads as an SM
    // holds or one of more (256 units of 800 candidates: 76.5 -> 71 us; 1024 units, several waves: 196 -> 198; 384
    // re-positioned units of 593, of whose CTAs an SM holds two: 89.6 in one launch, 78.5 in two).  Larger steps keep the two
    // launches, where a unit is selected once and the copies run at the copy rate.  So do batches of several requests on the tensor
    // cores: in one launch most small ones would be shorter (140 steps of 2 to 8 requests on 1 to 12 layers: 1.03 times as fast, up to
    // 1.12; 4 requests on 3 x 8 units 38.9 us, 36.0), but not those of few long units, each selected again by several CTAs of 512
    // threads (5 requests on 8 units of 2239 candidates 47.1 us, 50.5), and no line between them has been drawn.  A single request
    // takes the one launch however it was scored (prompts of more than 512 rows per KV head, 16 steps of 1 to 8 layers: 2 to 12 %
    // shorter, 7 x 4 units of 751 candidates 47.9 -> 42.9 us; 40 causal ones of 8 to 1500 rows 1 to 14 %).
    const int threads = max(kCompactThreads, pick::threads_for(max_n));
    const bool small = threads == kCompactThreads;
    const int most = (bv.max_budget + kMinRowsPerCta - 1) / kMinRowsPerCta, least = (bv.max_budget + kMaxRowsPicked - 1) / kMaxRowsPicked;
    const int blocks = units > 0 ? max(least, (int)min((int64_t)most, (small ? 2 : 1) * sms / units)) : 0;
    const bool two_launches = bv.batch > 1 && score_tc_supported(ctx);
    const auto wave = [&]() { return (small ? picks_per_sm(ctx, mv, pick::items_for(max_n)) : 1) * sms; };
    if (blocks == 0 || two_launches || max_n > kPickThreads * 8 || units * blocks > wave()) {
        const cudaError_t e = launch_select(ctx, scores, bv, kept_idx, out_len, stream);
        return e != cudaSuccess ? e : launch_compact(ctx, kept_idx, out_len, cache_k, cache_v, cache_pos, chunk_k, chunk_v,
                                                     chunk_pos, bv, out_k, out_v, out_pos, stream);
    }
    ctx.launches += 1;
    const CompactTensors t{cache_k, cache_v, chunk_k, chunk_v, out_k, out_v, cache_pos, chunk_pos, out_pos};
    return by_rotation(mv, [&](auto rope, auto elems) {
        constexpr int kRope = decltype(rope)::value, kElems = decltype(elems)::value;
        return launch_chained(pick::items_for(max_n) == 4 ? select_compact_kernel<kRope, kElems, 4> : select_compact_kernel<kRope, kElems, 8>,
                              dim3(blocks, heads, bv.batch), dim3(threads), 0, stream,
                              mv, bv, scores, kept_idx, out_len, t, (bv.max_budget + blocks - 1) / blocks, ctx.d_status);
    });
}

}  // namespace finch
