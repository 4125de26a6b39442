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

#include "finch_internal.cuh"

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

// Plain copies.  A thread keeps its piece of the row and walks the rows 256 / pieces apart.
__device__ __forceinline__ void copy_rows(const RowMap &m, const int *src_idx, int rows, int pieces) {
    constexpr int kBatch = 8;
    const int step = kCompactThreads / pieces, r0 = threadIdx.x / pieces, off = (threadIdx.x - r0 * pieces) * 16;
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
                                            const float2 *rope_table) {
    constexpr int kBatch = 4;
    const int half = d / 2, pieces = d * elem_bytes / 16 / (kSplit ? 2 : 1);
    const int step = kCompactThreads / pieces, r0 = threadIdx.x / pieces, piece = threadIdx.x - r0 * pieces;
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

// ROPE 0: bit-for-bit copies; 1 / 2: K rows re-positioned, pairs (t, t + d/2) / (2t, 2t + 1).
template <int ROPE, int kElems>
__global__ void __launch_bounds__(kCompactThreads)
compact_kernel(ModelView mv, BatchView bv, const int *kept_idx, const int *out_len, TensorView cache_k,
               TensorView cache_v, const int *cache_pos, TensorView chunk_k, TensorView chunk_v, const int *chunk_pos,
               TensorView out_k, TensorView out_v, int *out_pos, int rows_per_cta, int *status) {
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
    const bool leader = kvh == group * mv.kvpg;  // the group's positions are written by its first KV head's CTA

    if (threadIdx.x < rows) {
        int j = kept_idx[unit_off + i0 + threadIdx.x];
        // with rotation a distance beyond the table (only possible when out_len exceeds the candidate count) is refused
        if (j < 0 || j >= u.N || (ROPE && abs(i0 + (int)threadIdx.x - j) >= mv.rope_rows)) {
            atomicOr(status, FINCH_DEV_BAD_INDEX);
            j = -1;
        } else if (leader) {
            out_pos[unit_off + i0 + threadIdx.x] = j < u.c ? cache_pos[unit_off + j] : chunk_pos[u.chunk0 + j - u.c];
        }
        src_idx[threadIdx.x] = j;
    }
    __syncthreads();

    const int pieces = mv.d * mv.elem_bytes / 16;  // 16-byte pieces per row
    const RowMap k_rows(u, kvh, i0, mv.elem_bytes, cache_k, chunk_k, out_k);
    if (ROPE)
        rotate_rows<kElems, ROPE == 1>(k_rows, src_idx, rows, i0, mv.d, mv.elem_bytes, mv.rope_table);
    else
        copy_rows(k_rows, src_idx, rows, pieces);
    copy_rows(RowMap(u, kvh, i0, mv.elem_bytes, cache_v, chunk_v, out_v), src_idx, rows, pieces);
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
    const bool f32 = mv.elem_bytes == 4;
    auto kernel = compact_kernel<0, 8>;
    if (mv.rope_theta > 0.f && mv.rope_pairing == 0) kernel = f32 ? compact_kernel<1, 4> : compact_kernel<1, 8>;
    if (mv.rope_theta > 0.f && mv.rope_pairing == 1) kernel = f32 ? compact_kernel<2, 4> : compact_kernel<2, 8>;
    return launch_chained(kernel, grid, dim3(kCompactThreads), 0, stream, mv, bv, kept_idx, out_len, cache_k, cache_v,
                          cache_pos, chunk_k, chunk_v, chunk_pos, out_k, out_v, out_pos, rows, ctx.d_status);
}

}  // namespace finch
