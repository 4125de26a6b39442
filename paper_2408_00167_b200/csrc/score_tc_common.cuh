// Pieces shared by the tensor-core scoring kernels: tile geometry, the candidate view, the packed fp32 arithmetic of
// the two sweeps (row log-sum-exp, column sums), the merge of partial row statistics and the TMA tensor maps.
#pragma once

#include <limits.h>

#include "finch_internal.cuh"
#include "sm100_ptx.cuh"

namespace finch {
namespace tc {

using namespace ptx;

constexpr int kRows = 128;       // rows per operand tile = MMA M
constexpr int kRowPad = 8;       // a query head's prompt rows are padded to this many (the swizzle's 8-row group)
constexpr int kMaxRows = 512;    // padded query rows resident at a time: four query tiles
constexpr int kQTiles = kMaxRows / kRows;
constexpr int kGroups = 4;       // softmax groups of four warps; each owns one accumulator of 128 tensor-memory columns
constexpr int kMaxStages = 6;    // key-tile ring
constexpr int kSumBufs = 8;      // column-sum hand-over buffers, one per accumulator in flight
constexpr int kCtlWarps = 4;     // producer, MMA issuer, statistics warp, column-sum warp or second MMA issuer
constexpr int kSoftmaxWarps = 16;
constexpr int kTcThreads = (kCtlWarps + kSoftmaxWarps) * 32;
constexpr int kBigBox = 64;      // query rows per TMA box where a head has that many; kRowPad-row boxes otherwise
constexpr int kPlanBoundsInts = 1024;  // room for the per-CTA item bounds in the scratch (grid + 1 <= this)
constexpr int kSlabBytes = kRows * 128;  // a 64-element (128-byte) wide slab of a 128-row tile
constexpr int kSmemLimit = 232448;       // 227 KiB per CTA

struct KeyTile {
    int is_chunk;  // which tensor the rows come from
    int row0;      // first token row inside that packed tensor
    int j0;        // candidate index of the tile's first row
    int valid;     // rows of the tile that are candidates (1..128)
};

__device__ __forceinline__ int n_key_tiles(const UnitInfo &u) { return (u.c + kRows - 1) / kRows + (u.m + kRows - 1) / kRows; }

__device__ __forceinline__ KeyTile key_tile(const UnitInfo &u, int t) {
    const int tc = (u.c + kRows - 1) / kRows;
    KeyTile k;
    if (t < tc) {
        k.is_chunk = 0;
        k.row0 = u.cache0 + t * kRows;
        k.j0 = t * kRows;
        k.valid = min(kRows, u.c - t * kRows);
    } else {
        const int tt = t - tc;
        k.is_chunk = 1;
        k.row0 = u.chunk0 + tt * kRows;
        k.j0 = u.c + tt * kRows;
        k.valid = min(kRows, u.m - tt * kRows);
    }
    return k;
}

// The query rows of a scoring unit (layer, KV head, request): its query heads one after the other, each head's prompt
// rows padded to a multiple of 8.  Row r is prompt row r % rp of head r / rp.  Units of more than kMaxRows rows are
// worked on in chunks of kMaxRows (a row's softmax does not depend on the other rows).
//
// First sweep (a row per tensor-memory lane): row r of the chunk is lane r % 128 of query tile r / 128.  A warp only
// reaches the 32 lanes of its own quarter, so a last tile of at most 64 (32) rows would leave two (three) of the four
// schedulers idle: it is loaded twice (four times), `span` rows apart, and the copies share the columns.
// Second sweep (a key per lane, rows along the columns): an accumulator holds one key tile against a block of at most
// 128 rows (n_st blocks of `width`), or, for at most 64 rows, two key tiles side by side (kt = 2).
struct Rows {
    int n_q, rp;
    int r0, rows;         // the chunk's first padded row, its padded rows
    int n_qt, span;       // query tiles; rows of the last tile that are not copies (32, 64 or 128)
    int kt, n_st, width;  // key tiles per accumulator, accumulators per key tile, columns per key tile (multiple of 16)
};
__host__ __device__ inline int padded_rows(int n_q, int heads) { return heads * ((n_q + kRowPad - 1) / kRowPad * kRowPad); }
__device__ __forceinline__ Rows make_rows(int n_q, int heads, int chunk) {
    Rows r;
    r.n_q = n_q;
    r.rp = (n_q + kRowPad - 1) / kRowPad * kRowPad;
    r.r0 = chunk * kMaxRows;
    r.rows = max(0, min(kMaxRows, heads * r.rp - r.r0));
    r.n_qt = (r.rows + kRows - 1) / kRows;
    const int last = r.rows - (r.n_qt - 1) * kRows;
    r.span = last <= 32 ? 32 : (last <= 64 ? 64 : 128);
    const int cols = (r.rows + 15) & ~15;
    r.kt = cols <= 64 ? 2 : 1;
    r.n_st = (cols + kRows - 1) / kRows;
    r.width = r.n_st > 1 ? ((cols / r.n_st + 15) & ~15) : cols;
    return r;
}
// Is padded row r of the chunk a prompt row?
__device__ __forceinline__ bool row_live(const Rows &r, int row) { return row < r.rows && (r.r0 + row) % r.rp < r.n_q; }

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed pairs of fp32 (sm_100 executes these as one instruction on the FMA pipe).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float4 lds128(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// exp2 of a pair.  (A degree-5 polynomial on the FMA pipe for an eighth to a third of the pairs makes the loops alone 8
// to 15 % shorter, but not the calls, in loops of seconds under the 1000 W power limit: 32 layers x 8 heads x 4096 candidates x 512 rows, whole step, 0.452 ms without, 0.453 with an eighth, 0.465 with
// a quarter.)
__device__ __forceinline__ uint64_t exp2_pair(uint64_t x2) {
    float x0, x1;
    unpack2(x2, x0, x1);
    return pack2(ex2(x0), ex2(x1));
}

// First sweep: fold NC columns (keys) of one accumulator row into the row's running (reference, sum of exp2).
// The reference is the maximum of the row's first chunk, not the running maximum: any reference works as long as
// the sum stays finite, and skipping the per-element maximum saves a quarter of the instructions.  If the sum
// overflows (a later logit more than ~2^7 base-2 units above the reference, or many nearly that far) the reference
// moves up and the chunk is redone.  Columns at or beyond nv hold no key and count nothing.
//
// The rare parts (a tile's ragged end, a row's first chunk) sit behind warp-uniform branches with an empty asm in them, which
// asks for a branch in place of predication: whole and ragged tiles then cost what they contain.
__device__ __forceinline__ void keep_branch() { asm volatile("" ::: "memory"); }
template <int NC>
__device__ __forceinline__ void mask_tail(uint32_t (&r)[NC], int nv) {
    if (__any_sync(0xffffffffu, nv < NC)) {
        keep_branch();
#pragma unroll
        for (int e = 0; e < NC; ++e)
            if (e >= nv) r[e] = 0xff800000u;  // -inf
    }
}
template <int NC>
__device__ __forceinline__ float chunk_max(const uint32_t (&r)[NC]) {
    float m = __uint_as_float(r[0]);
#pragma unroll
    for (int e = 1; e < NC; ++e) m = fmaxf(m, __uint_as_float(r[e]));
    return m;
}
// The bare sum of 32 columns against a reference (negm = -reference * scale2), in two pairs of partial sums.
template <int NC>
__device__ __forceinline__ void lse_sum(const uint32_t (&r)[NC], float scale2, float negm, uint64_t &acc0, uint64_t &acc1) {
    const uint64_t s2 = pack2(scale2, scale2), n2 = pack2(negm, negm);
#pragma unroll
    for (int e = 0; e < NC; e += 4) {
        acc0 = add2(acc0, exp2_pair(fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), s2, n2)));
        acc1 = add2(acc1, exp2_pair(fma2(pack2(__uint_as_float(r[e + 2]), __uint_as_float(r[e + 3])), s2, n2)));
    }
}
__device__ __forceinline__ float sum_of(uint64_t acc0, uint64_t acc1) {
    float a0, a1, a2, a3;
    unpack2(acc0, a0, a1);
    unpack2(acc1, a2, a3);
    return (a0 + a1) + (a2 + a3);
}
template <int NC>
__device__ __forceinline__ void lse_chunk(uint32_t (&r)[NC], int nv, bool live, float scale2, float &m_raw, float &z) {
    mask_tail(r, nv);
    if (__any_sync(0xffffffffu, m_raw == -INFINITY && live)) {
        keep_branch();
        const float cmax = chunk_max(r);
        if (m_raw == -INFINITY) m_raw = cmax;
    }
    auto sum = [&]() -> float {
        uint64_t acc0 = 0, acc1 = 0;  // +0.0f bit patterns
        lse_sum(r, scale2, -(m_raw * scale2), acc0, acc1);
        return sum_of(acc0, acc1);
    };
    const float zn = z + sum();
    if (__any_sync(0xffffffffu, !(zn <= 3.0e38f) && live)) {
        keep_branch();
        // Overflow (inf or NaN) on some lane: it moves its reference up and redoes the chunk.  The new reference must cover
        // the chunk's largest logit and what has been summed so far (z = 2^e * [1, 2) against the old reference, e from
        // z's exponent field), so that the redone sum is at most 1 + NC.  The factor between the two references (the
        // same rounded products the chunks subtract) is applied in two halves, since z may be near 2^127 while the
        // factor is below the smallest normal number.
        if (!(zn <= 3.0e38f) && live) {
            const float lift = (float)(((__float_as_int(z) >> 23) & 0xff) - 126);
            const float m_new = fmaxf(chunk_max(r), fmaf(lift, __frcp_rn(scale2), m_raw));
            const float half_d = 0.5f * (__fmul_rn(m_raw, scale2) - __fmul_rn(m_new, scale2));
            z = (z * ex2(half_d)) * ex2(half_d);
            m_raw = m_new;
            z += sum();
        } else if (live) {
            z = zn;
        }
    } else if (live) {
        z = zn;
    }
}

// Second sweep: add to (c0, c1) the weights exp2(s * scale2 - ref_r) * w_r of NC columns (prompt rows) of one accumulator
// row (a key).  The statistics are staged in pairs of rows, (-ref_a, -ref_b, w_a, w_b), so that one 128-bit load feeds
// two packed operations.
// Masked variant: lim2 holds, per pair of rows, how many candidates each row attends to; this thread's key has
// candidate index j and counts for a row only if j is below that row's number.
template <int NC, bool MASK>
__device__ __forceinline__ void colsum_chunk(const uint32_t (&r)[NC], float scale2, uint32_t sm4, float &c0, float &c1,
                                             const int2 *lim2, int j) {
    const uint64_t s2 = pack2(scale2, scale2);
    uint64_t acc = pack2(c0, c1);
#pragma unroll
    for (int e = 0; e < NC; e += 2) {
        const float4 s4 = lds128(sm4 + (e / 2) * 16);  // two prompt rows: (-ref_a, -ref_b, w_a, w_b)
        uint64_t x = fma2(pack2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), s2, pack2(s4.x, s4.y));
        if (MASK) {
            float x0, x1;
            unpack2(x, x0, x1);
            const int2 l2 = lim2[e / 2];
            x0 = j < l2.x ? x0 : -INFINITY;  // exp2(-inf) = 0: the row does not see this key
            x1 = j < l2.y ? x1 : -INFINITY;
            x = pack2(x0, x1);
        }
        acc = fma2(exp2_pair(x), pack2(s4.z, s4.w), acc);
    }
    unpack2(acc, c0, c1);
}

// ---- merging partial row statistics.  A part is (reference, sum of exp2 against that reference), both in base-2
// logit units; parts are folded in a fixed order into a running (M, Z), then turned into the pair the column
// sweep uses: weights are exp2(s2 - R) * w with R = M + floor(log2 Z) and w = 2^floor(log2 Z) / Z in (1/2, 1], so
// the exponent never exceeds a few units whatever reference the parts were summed against.
__device__ __forceinline__ float2 normal_part(float2 pm) {
    // A part's sum can be as large as 2^127 against a reference that far below its largest logit: move the sum's
    // exponent into the reference, so that no factor below leaves the fp32 range.  A part that saw none of the row's
    // logits (sum 0; any other sum is at least 1, a normal number) becomes (-inf, 0).
    const int bits = __float_as_int(pm.y);
    if (!(pm.y > 0.f)) return make_float2(-INFINITY, 0.f);
    return make_float2(pm.x + (float)(((bits >> 23) & 0xff) - 127), __int_as_float((bits & 0x007fffff) | 0x3f800000));
}
template <int N>
__device__ __forceinline__ void merge_parts(const float2 (&raw)[N], float &M, float &Z) {
    float2 part[N];
    float nm = M;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        part[i] = normal_part(raw[i]);
        nm = fmaxf(nm, part[i].x);
    }
    if (nm == -INFINITY) return;
    Z *= ex2(M - nm);
#pragma unroll
    for (int i = 0; i < N; ++i) Z += part[i].y * ex2(part[i].x - nm);
    M = nm;
}
// One more part with sum 1 whose reference is a natural-log value (the keys a row attends to besides the candidates).
__device__ __forceinline__ void merge_self_term(float lse_nat, float &M, float &Z) {
    const float px = lse_nat * kLog2e;
    if (px > -INFINITY) {
        const float nm = fmaxf(M, px);
        Z = Z * ex2(M - nm) + ex2(px - nm);
        M = nm;
    }
}
// (M, Z) -> the row's natural-log sum-exp, and (-R, w).  A row that attends to nothing (Z = 0) weighs nothing: -inf and
// (0, 0).
__device__ __forceinline__ float merged_lse(float M, float Z) { return Z > 0.f ? (M + log2f(Z)) * kLn2 : -INFINITY; }
__device__ __forceinline__ float2 merged_pair(float M, float Z) {
    if (!(Z > 0.f)) return make_float2(0.f, 0.f);
    // Z = 2^k * [1, 2) (a sum of terms in [1, 2) times factors <= 1, the largest of them 1)
    const int zbits = __float_as_int(Z);
    const int k = ((zbits >> 23) & 0xff) - 127;
    const float w = __fdividef(1.0f, __int_as_float((zbits & 0x007fffff) | 0x3f800000));
    return make_float2(-(M + (float)k), w);
}

// rows 2k and 2k+1 share one float4: (-ref_2k, -ref_2k+1, w_2k, w_2k+1)
__device__ __forceinline__ void stage_row(float2 *stats, int row, float2 v) {
    float *f = (float *)stats + (row >> 1) * 4 + (row & 1);
    f[0] = v.x;
    f[2] = v.y;
}

// ------------------------------------------------------------------------------------------------ host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        return (EncodeTiledFn)p;
    }();
    return fn;
}

// [layers][heads][tokens][d] bf16 view -> 4-D tensor map with a (64 elements x box_rows) box, 128-byte swizzle.
inline bool make_map(CUtensorMap *map, const TensorView &t, int d, int64_t tokens, int heads, int layers, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn || !t.ptr || tokens <= 0) return false;
    const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)tokens, (cuuint64_t)heads, (cuuint64_t)layers};
    const cuuint64_t strides[3] = {(cuuint64_t)t.stride_tok * 2, (cuuint64_t)t.stride_head * 2,
                                   (cuuint64_t)t.stride_layer * 2};
    for (int i = 0; i < 3; ++i)
        if (strides[i] == 0 || strides[i] % 16 || strides[i] >= (1ull << 40)) return false;
    const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<char *>(t.ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace finch
