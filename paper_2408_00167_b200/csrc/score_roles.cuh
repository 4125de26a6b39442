// The roles of a tensor-core scoring CTA, shared by the one-kernel and the two-launch path.  A kernel walks a list of
// segments -- (sweep, unit, key-tile range) -- and every role walks the same list with the same running counters, so
// barrier phases stay in step without any further handshake.
//
//   Producer     one warp: query tiles (resident while the unit stays the same) and the ring of key tiles, by TMA.
//   PadCleaner   the producer itself or a warp of its own: zeroes pad rows of the queries that hold other rows.
//   Issuer       one warp: tcgen05.mma into four accumulators of 128 tensor-memory columns in turn; in the one-kernel path two
//                warps, every second accumulator each, for units of one query tile.
//   Softmax      four groups of four warps (a warp per lane quarter): accumulator number A belongs to group A % 4.  A
//                scheduler holds one warp of each group, so three of them compute while one waits for its refill.
//   SumWriter    one warp: adds the row blocks' column sums of a key (second sweep) and writes the scores.  Where two warps
//                issue there is one block, and the softmax warps write.
//
// What bounds it, for units of several query tiles: two exponentials per logit, 1024 clocks of the special-function unit per 128 x 128 logits and sweep,
// and the chip's power limit (large calls run at 1.70 to 1.85 GHz).  Measured on the loops alone (accumulators refilled by
// MMAs, no loads): 1150 clocks per accumulator in the first sweep and 1210 in the second.  Bookkeeping counts: every
// instruction between two accumulators is paid by sixteen warps, so what can be is worked out per segment, ragged ends
// and overflow repairs leave for a path out of line, and barriers are addressed by their shared-memory address.
#pragma once

#include "score_tc_common.cuh"

namespace finch {
namespace tc {

struct Cta {  // shared memory of the CTA
    uint8_t *q_res, *ring;
    uint64_t *q_raw;                   // [kQTiles] a query tile has landed, its pad rows are still to be cleared
    uint64_t *q_full, *q_free;         // [kQTiles] query tile has landed / its last MMAs are complete
    uint64_t *full, *empty;            // [kMaxStages] key ring
    uint64_t *acc_full, *acc_empty;    // [kGroups] accumulators
    uint64_t *stats_ready;             // [2] row statistics of a second-sweep segment are staged
    uint64_t *sum_full, *sum_empty;    // [kSumBufs] column sums handed to the writer
    uint64_t *parts_ready;             // the cluster's CTAs have written their partial row statistics
    uint32_t *tmem_slot;
    volatile int *abort_flag;
    int *a_count;                      // softmax warps through a first-sweep segment (counts up for ever)
    float *sums;                       // [kSumBufs][2][kRows]
    float2 *stats;                     // [2][rows] (-ref, weight), pairs of rows interleaved
    int *limits;                       // [2][rows] visible candidates per row (masked variant) ..
    int2 *bounds;                      // [2][rows / 16] .. and the least and the most of every 16 rows
    int q_slab;                        // bytes of one 64-element slab of the resident queries
    int stages;
    int q_tiles;                       // query tiles the shared memory holds
    int rows_alloc;                    // rows of a statistics buffer (a multiple of 128)
};

constexpr int kBarBytes = 512;
constexpr int kSumBytes = kSumBufs * 2 * kRows * 4;
constexpr int cta_smem(int tile_bytes, int q_tiles, int rows_alloc, int stages, bool mask) {
    return 1024 + (q_tiles + stages) * tile_bytes + kBarBytes + kSumBytes + 2 * rows_alloc * 8 +
           (mask ? 2 * rows_alloc * 4 + rows_alloc : 0);
}

__device__ __forceinline__ Cta cta_layout(uint8_t *raw, int tile_bytes, int q_tiles, int rows_alloc, int stages) {
    Cta c;
    uint8_t *s = (uint8_t *)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
    c.q_res = s;
    c.q_slab = q_tiles * kSlabBytes;
    c.q_tiles = q_tiles;
    c.rows_alloc = rows_alloc;
    c.stages = stages;
    c.ring = s + q_tiles * tile_bytes;
    uint8_t *aux = c.ring + stages * tile_bytes;
    uint64_t *b = (uint64_t *)aux;
    c.q_full = b, b += kQTiles;
    c.q_free = b, b += kQTiles;
    c.full = b, b += kMaxStages;
    c.empty = b, b += kMaxStages;
    c.acc_full = b, b += kGroups;
    c.acc_empty = b, b += kGroups;
    c.stats_ready = b, b += 2;
    c.sum_full = b, b += kSumBufs;
    c.sum_empty = b, b += kSumBufs;
    c.q_raw = b, b += kQTiles;
    c.parts_ready = b, b += 1;
    c.tmem_slot = (uint32_t *)b;
    c.abort_flag = (volatile int *)(c.tmem_slot + 1);
    c.a_count = (int *)(c.tmem_slot + 2);
    c.sums = (float *)(aux + kBarBytes);
    c.stats = (float2 *)(aux + kBarBytes + kSumBytes);
    c.limits = (int *)(c.stats + 2 * rows_alloc);
    c.bounds = (int2 *)(c.limits + 2 * rows_alloc);
    return c;
}

// Barriers and tensor memory (all 512 columns); ends with the CTA in step.  stats_arrivals: arrivals per staging.
// cluster: CTAs that exchange row statistics through each other's shared memory (1: none).
// issuers: MMA issuers that share the key and query tiles.
__device__ __forceinline__ uint32_t cta_setup(const Cta &c, int stats_arrivals, int cluster = 1, int issuers = 1) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < kQTiles; ++i) {
            mbar_init(&c.q_raw[i], 1);
            mbar_init(&c.q_full[i], 1);
            mbar_init(&c.q_free[i], issuers);
        }
        for (int i = 0; i < kMaxStages; ++i) {
            mbar_init(&c.full[i], 1);
            mbar_init(&c.empty[i], issuers);
        }
        for (int i = 0; i < kGroups; ++i) {
            mbar_init(&c.acc_full[i], 1);
            mbar_init(&c.acc_empty[i], 4);
        }
        for (int i = 0; i < 2; ++i) mbar_init(&c.stats_ready[i], stats_arrivals);
        for (int i = 0; i < kSumBufs; ++i) {
            mbar_init(&c.sum_full[i], 4);
            mbar_init(&c.sum_empty[i], 1);
        }
        mbar_init(c.parts_ready, cluster * kSoftmaxWarps);
        *c.abort_flag = 0;
        *c.a_count = 0;
        fence_barrier_init();
    }
    if (threadIdx.x / 32 == 1) {
        tmem_alloc(c.tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    if (cluster > 1) cluster_arrive();  // the barriers are initialised: waited for ahead of the first remote arrival
    tc_fence_after();
    return *c.tmem_slot;
}

// Common epilogue: everyone meets here, also after a timed-out wait.  The single-thread roles bring their warps back
// together first: the CTA barrier must be executed by whole warps.
// left: this warp has been through both cluster barriers but the last wait.
__device__ __forceinline__ void cta_teardown(const Cta &c, uint32_t tmem, int *status, int cluster = 1, bool left = false) {
    __syncwarp();
    if (cluster > 1 && !left) {
        cluster_wait();
        cluster_arrive();
    }
    tc_fence_before();
    __syncthreads();
    if (cluster > 1) cluster_wait();  // the neighbours have read this CTA's shared memory
    if (threadIdx.x == 0 && *c.abort_flag) atomicOr(status, FINCH_DEV_TIMEOUT);
    if (threadIdx.x / 32 == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// The resident query tiles as a ring: a load of n tiles takes the next n, all behind one another, so that the queries of the
// next unit can arrive while the MMAs still read those of the current one wherever both fit.
struct TileRing {
    int tiles, pos = 0;
    __device__ int take(int n) {
        if (pos + n > tiles) pos = 0;
        const int base = pos;
        pos += n;
        return base;
    }
};

// ------------------------------------------------------------------------------------------------ producer
// Pad rows that lie inside the query tensor hold whatever comes behind the request's own rows: the next request's, or rows that
// another call uses.  (Behind the tensor's last row the copies deliver zeros.)  They weigh nothing, but a NaN among them, or a
// logit whose exponential overflows, would still reach this request's sums: they are cleared between the copy and the MMAs.
__device__ __forceinline__ bool pads_hold_rows(const UnitInfo &u, const Rows &R, int total_q) {
    return R.rp != R.n_q && u.q0 + R.n_q < total_q;
}

// Run by a whole warp: clears the pad rows of query tiles as they land and hands them to the MMAs.  In the two-launch kernels
// by a warp of its own, so that the producer runs on to the next unit's queries (31 requests of up to 3 rows and 56 candidates
// on 29 x 8 units: 610 us with the producer waiting for every unit's rows, 412 with this).
template <int D>
struct PadCleaner {
    static constexpr int kSlabs = D / 64;
    const Cta &c;
    uint32_t ph = 0;  // bit per query tile: parity of its next q_raw phase
    __device__ bool clear(const Rows &R, int base) {
        const int pads = R.rp - R.n_q, lane = threadIdx.x & 31;  // at most seven rows of 8 pieces per head and slab
        for (int qb = 0; qb < R.n_qt; ++qb) {
            const int tile = base + qb, r0 = R.r0 + qb * kRows, r1 = min(r0 + kRows, R.r0 + R.rows);  // padded rows of the unit
            if (!__all_sync(0xffffffffu, mbar_wait(&c.q_raw[tile], ph >> tile & 1u, c.abort_flag))) return false;
            ph ^= 1u << tile;
            // (the copies of a short last tile need no clearing, their lanes are skipped)
            for (int h = r0 / R.rp; h * R.rp < r1; ++h)
                for (int i = lane; i < pads * 8 * kSlabs; i += 32) {
                    const int s = i / (pads * 8), k = i - s * pads * 8, r = h * R.rp + R.n_q + k / 8;
                    if (r >= r0 && r < r1)
                        *(uint4 *)(c.q_res + s * c.q_slab + (tile * kRows + r - r0) * 128 + k % 8 * 16) = uint4{0, 0, 0, 0};
                }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.q_full[tile]);
        }
        return true;
    }
};

// Run by a whole warp.  OWN_WARP: the PadCleaner is a warp of its own; FIRST_SWEEP: the queries are (also) for the first sweep.
template <int D, bool OWN_WARP, bool FIRST_SWEEP>
struct Producer {
    static constexpr int kSlabs = D / 64, kTileBytes = kSlabs * kSlabBytes;
    const Cta &c;
    const CUtensorMap *q_big, *q_small, *cache, *chunk;
    int heads;    // query heads per unit
    int total_q;  // query rows of the packed tensor
    int key_shift = 0;  // units that share a KV head, as a power of two
    PadCleaner<D> cleaner{c};
    int st = 0, ph = 0, kcnt = 0;
    uint32_t q_used = 0, q_ph = 0;  // bit per query tile: loaded before / parity of its next q_free phase

    __device__ __forceinline__ bool agree(bool ok) { return __all_sync(0xffffffffu, ok); }
    __device__ bool load_key_tile(const UnitInfo &u, int t) {
        const int stage = st, p = ph;
        if (++st == c.stages) {
            st = 0;
            ph ^= 1;
        }
        // a producer a ring ahead of the MMAs polls rarely: its tests share a queue with the special-function unit
        if (!agree(mbar_wait_relaxed(&c.empty[stage], p ^ 1, c.abort_flag, 500))) return false;
        const KeyTile kt = key_tile(u, t);
        const CUtensorMap *m = kt.is_chunk ? chunk : cache;
        if (elect_one()) {
            mbar_expect_tx(&c.full[stage], kTileBytes);
            for (int s = 0; s < kSlabs; ++s)
                tma_load_4d(c.ring + stage * kTileBytes + s * kSlabBytes, m, &c.full[stage], s * 64, kt.row0, u.G >> key_shift, u.l);
        }
        ++kcnt;
        return true;
    }
    // The n padded rows from the unit's row r on to resident query tile `tile` (and its copies, `span` rows apart).  A lane
    // takes eight rows of one slab and copy, or issues the box of 64 rows that begins with them; no box leaves its head.  One
    // lane that walks the boxes, up to 32 with a division each, takes a microsecond for a unit of few rows (13 requests of up
    // to 9 rows on 19 x 8 units: 124 us, 109 with the lanes).
    __device__ __forceinline__ void load_tile(const UnitInfo &u, const Rows &R, int r, int n, int span, int copies, int tile,
                                              uint64_t *bar) {
        const int lane = threadIdx.x & 31, s = lane >> 4, shift = span == 128 ? 4 : (span == 64 ? 3 : 2);
        const int copy = (lane & 15) >> shift, i = lane & ((1 << shift) - 1);
        const int row = r + i * kRowPad, h = row / R.rp, start = max(r, h * R.rp), end = min(r + n, (h + 1) * R.rp);
        const int big_rows = (end - start) & ~(kBigBox - 1), at = row - start;  // boxes of 64 rows first, then of 8
        if (elect_one()) mbar_expect_tx(bar, n * copies * 128 * kSlabs);
        __syncwarp();
        if (s < kSlabs && copy < copies && row < r + n && (at >= big_rows || at % kBigBox == 0))
            tma_load_4d(c.q_res + s * c.q_slab + (tile * kRows + copy * span + i * kRowPad) * 128, at < big_rows ? q_big : q_small,
                        bar, s * 64, u.q0 + row - h * R.rp, u.G * heads + h, u.l);
        __syncwarp();
    }
    // The unit's query tiles into the ring's tiles base .., one at a time: a tile may be overwritten once the last MMAs on
    // its old contents are complete, while the MMAs on the tiles behind it still run.
    __device__ __forceinline__ bool load_queries(const UnitInfo &u, const Rows &R, int base) {
        const bool raw = pads_hold_rows(u, R, total_q);  // a PadCleaner stands between the copies and the MMAs
        uint64_t *const landed = raw ? c.q_raw : c.q_full;
        for (int qb = 0; qb < R.n_qt; ++qb) {
            const int tile = base + qb, r = qb * kRows, n = min(kRows, R.rows - r), span = qb < R.n_qt - 1 ? kRows : R.span;
            const int copies = FIRST_SWEEP ? kRows / span : 1;  // the second sweep reads the rows along the columns: once
            if (q_used >> tile & 1u) {
                if (!agree(mbar_wait(&c.q_free[tile], q_ph >> tile & 1u, c.abort_flag))) return false;
                q_ph ^= 1u << tile;
            }
            q_used |= 1u << tile;
            load_tile(u, R, R.r0 + r, n, span, copies, tile, landed + tile);
        }
        return !raw || OWN_WARP || cleaner.clear(R, base);
    }
    // One segment; base: the ring tiles its queries are to be loaded into, or -1: they are resident.
    __device__ bool segment(const UnitInfo &u, const Rows &R, int t0, int t1, int base) {
        // the segment's first key tile goes first: its ring stage is free before the query tiles are
        if (!load_key_tile(u, t0)) return false;
        if (base >= 0 && !load_queries(u, R, base)) return false;
        for (int t = t0 + 1; t < t1; ++t)
            if (!load_key_tile(u, t)) return false;
        return true;
    }
    // No copy may still be in flight when the CTA retires: wait (bounded) for the last loads issued.  (A query tile's
    // q_full phases alternate with its q_free phases: q_ph has the parity of the last load.)
    __device__ void drain() {
        for (int i = 0; i < kQTiles; ++i)
            if (q_used >> i & 1u) mbar_wait(&c.q_full[i], q_ph >> i & 1u, c.abort_flag);
        for (int i = max(0, kcnt - c.stages); i < kcnt; ++i) mbar_wait(&c.full[i % c.stages], (i / c.stages) & 1, c.abort_flag);
    }
};

// ------------------------------------------------------------------------------------------------ MMA issuer
// Run by a whole warp: one elected lane issues, the others keep the control flow uniform (see elect_one).
//
// PAIR: two warps issue, for units of one query tile, every second accumulator (and its key tiles) each.  One warp needs 1300 clocks for
// the accumulator of a key tile even where nothing is late -- two barrier tests of 150 to 200 beside warps whose exponentials fill the
// queue that barriers share with them, 390 for the eight MMAs, 220 for the commits -- against 500 of MMAs and, for 64 rows, as
// many of exponentials.  (32 x 32 units of 8 key tiles x 64 rows 101 -> 98 us, of 11 x 80 rows 141 -> 131; 23 x 8 units of 16 tiles x 24
// rows, head_dim 64, 38.5 -> 31.3.)  With more query tiles the softmax warps are the slower side.  Both pass every key tile, and a stage is
// refilled when both have: a barrier's parity tells a phase from its neighbours only, so neither may fall two loads behind or ahead.
template <int D, bool PAIR = false>
struct Issuer {
    static constexpr int kSlabs = D / 64, kTileBytes = kSlabs * kSlabBytes;
    const Cta &c;
    uint32_t tmem, desc_hi, q_lo, ring_lo, q_slab;
    uint32_t A = 0;  // accumulators issued
    int st = 0, ph = 0;
    uint32_t q_ph = 0;  // bit per query tile: parity of its next q_full phase
    uint32_t half;      // PAIR: the accumulators this warp issues, odd or even

    __device__ Issuer(const Cta &cta, uint32_t tm, uint32_t h = 0) : c(cta), tmem(tm), half(h) {
        const uint64_t q = smem_desc_sw128(smem_u32(c.q_res)), r = smem_desc_sw128(smem_u32(c.ring));
        desc_hi = (uint32_t)(q >> 32);
        q_lo = (uint32_t)q;
        ring_lo = (uint32_t)r;
        q_slab = (uint32_t)c.q_slab >> 4;
    }
    // D = A B^T over head_dim; the operands differ in their descriptors' low words only (the 14-bit address field
    // cannot carry: shared memory ends below 2^18 bytes).
    __device__ __forceinline__ void mma(uint32_t d, uint32_t a_lo, uint32_t a_slab, uint32_t b_lo, uint32_t b_slab,
                                        uint32_t idesc) {
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
            const uint64_t a = ((uint64_t)desc_hi << 32) | (a_lo + (k / 4) * a_slab + (k % 4) * 2);
            const uint64_t b = ((uint64_t)desc_hi << 32) | (b_lo + (k / 4) * b_slab + (k % 4) * 2);
            if (elect_one()) {
                if (k == 0)
                    umma_bf16_first(d, a, b, idesc);
                else
                    umma_bf16_acc(d, a, b, idesc);
            }
        }
    }
    __device__ __forceinline__ void commit(uint64_t *bar) {
        if (elect_one()) umma_commit(bar);
    }
    __device__ __forceinline__ bool wait(uint64_t *bar, uint32_t parity) {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity, c.abort_flag));
    }
    __device__ __forceinline__ bool acquire() { return wait(&c.acc_empty[A & 3], ((A >> 2) & 1) ^ 1); }
    __device__ __forceinline__ uint32_t acc() const { return tmem + (A & 3) * kRows; }
    __device__ __forceinline__ void publish() {
        commit(&c.acc_full[A & 3]);
        ++A;
    }
    __device__ __forceinline__ void next_key_stage(bool read = true) {
        if (read)
            commit(&c.empty[st]);  // the stage may be refilled once these MMAs have read it
        else if (elect_one())
            mbar_arrive(&c.empty[st]);
        if (++st == c.stages) {
            st = 0;
            ph ^= 1;
        }
    }
    __device__ __forceinline__ bool landed(int tile) {
        const bool ok = wait(&c.q_full[tile], q_ph >> tile & 1u);
        q_ph ^= 1u << tile;
        return ok;
    }
    // First sweep: D = query tile x key tile^T, one accumulator per (key tile, query tile).  base: the queries' tiles in
    // the ring; reload: they are being loaded; release: no later segment uses this load.
    __device__ bool lse_segment(const Rows &R, int t0, int t1, int base, bool reload, bool release) {
        constexpr uint32_t idesc = idesc_bf16_f32(kRows, kRows);
        if (PAIR && reload && !landed(base)) return false;
        for (int t = t0; t < t1; ++t) {
            if (!wait(&c.full[st], ph)) return false;
            if (PAIR && (A & 1) != half) {  // the other issuer's
                ++A;
                next_key_stage(false);
                continue;
            }
            const uint32_t b_lo = ring_lo + (uint32_t)(st * (kTileBytes >> 4));
            for (int qb = 0; qb < R.n_qt; ++qb) {
                if (!acquire()) return false;
                if (!PAIR && reload && t == t0 && !landed(base + qb)) return false;
                tc_fence_after();
                mma(acc(), q_lo + (uint32_t)((base + qb) * (kRows * 128 >> 4)), q_slab, b_lo, kSlabBytes >> 4, idesc);
                publish();
                if (!PAIR && release && t == t1 - 1) commit(&c.q_free[base + qb]);
            }
            next_key_stage();
        }
        if (PAIR && release) commit(&c.q_free[base]);  // also where none of the segment's accumulators was this warp's
        return true;
    }
    // Second sweep: D = key tile x query rows^T.
    __device__ bool colsum_segment(const Rows &R, int t0, int t1, int base, bool reload, bool release) {
        const int cols = (R.rows + 15) & ~15;
        bool side = false;  // kt = 2: this key tile takes the right half of the accumulator
        if (PAIR && reload && !landed(base)) return false;
        for (int t = t0; t < t1; ++t) {
            const bool last = t == t1 - 1;
            if (!wait(&c.full[st], ph)) return false;
            if (PAIR && (A & 1) != half) {  // the other issuer's
                next_key_stage(false);
                if (R.kt == 1 || side || last) ++A;
                side = R.kt == 2 && !side;
                continue;
            }
            const uint32_t a_lo = ring_lo + (uint32_t)(st * (kTileBytes >> 4));
            int freed = 0, seen = 0;
            for (int s = 0; s < R.n_st; ++s) {
                if (!side && !acquire()) return false;
                const int row = s * R.width, n = min(R.width, cols - row), tiles = min(R.n_qt, (row + n + kRows - 1) / kRows);
                if (!PAIR && reload && t == t0)
                    for (; seen < tiles; ++seen)
                        if (!landed(base + seen)) return false;
                tc_fence_after();
                mma(acc() + (side ? kRows / 2 : 0), a_lo, kSlabBytes >> 4, q_lo + (uint32_t)((base * kRows + row) * 128 >> 4),
                    q_slab, idesc_bf16_f32(kRows, n));
                if (R.kt == 1 || side || last) publish();
                if (!PAIR && release && last) {
                    const int done = s == R.n_st - 1 ? R.n_qt : (row + n) / kRows;
                    for (; freed < done; ++freed) commit(&c.q_free[base + freed]);
                }
            }
            next_key_stage();
            side = R.kt == 2 && !side;
        }
        if (PAIR && release) commit(&c.q_free[base]);
        return true;
    }
};

// ------------------------------------------------------------------------------------------------ softmax warps
// The parts of the first sweep that are rarely needed, out of line so that the hot loops fit the instruction cache: n
// columns from taddr, of which this lane's row sees nl and the warp's rows at most nv.
template <bool MASK>
__device__ __noinline__ float2 lse_any(uint32_t taddr, int n, int nv, int nl, bool live, float scale2, float m, float z) {
#pragma unroll 1
    for (int cc = 0; cc < n && cc < nv; cc += 16) {
        uint32_t r[16];
        __syncwarp();
        tmem_ld_issue(taddr + cc, r);
        tmem_ld_wait(r);
        lse_chunk<16>(r, nl - cc, MASK ? live && nl - cc > 0 : live, scale2, m, z);
    }
    return make_float2(m, z);
}

template <bool MASK>
struct Softmax {
    const Cta &c;
    uint32_t tmem;         // this warp's lanes of the group's accumulator
    uint32_t full, empty;  // shared-memory addresses of its barriers
    float scale2;
    int lane, quarter, group, my_row;
    uint32_t A = 0;     // accumulators of all groups before this segment
    uint32_t mine = 0;  // accumulators this group has consumed
    uint32_t E = 0;     // accumulators of second-sweep segments before this one

    __device__ Softmax(const Cta &cta, uint32_t tm, float s2) : c(cta), scale2(s2) {
        const int warp = threadIdx.x / 32;
        lane = threadIdx.x & 31;
        quarter = warp & 3;  // tcgen05.ld reaches lanes 32 * (warp % 4) ..
        group = (warp - kCtlWarps) >> 2;
        my_row = quarter * 32 + lane;
        tmem = tm + ((uint32_t)(quarter * 32) << 16) + group * kRows;
        full = smem_u32(c.acc_full + group);
        empty = smem_u32(c.acc_empty + group);
    }
    // a wait's verdict is made warp-uniform so that a timeout takes the whole warp out
    __device__ __forceinline__ bool acquire() {
        if (!__all_sync(0xffffffffu, mbar_wait(full, mine & 1, c.abort_flag))) return false;
        ++mine;
        tc_fence_after();
        return true;
    }
    __device__ __forceinline__ void release() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(empty);
    }
    // Row of the chunk this thread owns in query tile qb (may lie beyond R.rows).
    __device__ __forceinline__ int row_of(const Rows &R, int qb) const {
        return qb * kRows + (qb == R.n_qt - 1 ? my_row % R.span : my_row);
    }
    // First sweep over key tiles [t0, t1).  live: bit qb, this thread's row of query tile qb is a prompt row; lim (masked
    // variant): candidates that row attends to.  Of four, two or one query tiles a group meets the same one throughout a
    // segment; of three all, in turn: their statistics then rotate through slot 0.  On return slot k holds (m, z) of
    // query tile (qb + k) % n_qt.
    struct RowStats {
        float m[3], z[3];
        int qb;   // query tile of slot 0
        int rel;  // position of the segment's first accumulator of this group: where its statistics are stored
    };
    __device__ __forceinline__ bool lse_segment(const UnitInfo &u, const Rows &R, int t0, int t1, uint32_t live,
                                                const int (&lim)[kQTiles], RowStats &st) {
        const int n_qt = R.n_qt, first = (group - A) & 3;  // this group's first accumulator of the segment
        st.rel = first;
        int qb = first % n_qt, t = t0 + first / n_qt;
        const int step = n_qt == 1 ? 4 : (n_qt == 2 ? 2 : 1);
        A += (t1 - t0) * n_qt;
        const int cache_tiles = (u.c + kRows - 1) / kRows, all_tiles = n_key_tiles(u);
        // tiles of fewer than 128 keys: the last of the cache and of the chunk
        const int nv_cache = u.c - (cache_tiles - 1) * kRows, nv_chunk = u.m - (all_tiles - cache_tiles - 1) * kRows;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            st.m[k] = -INFINITY;
            st.z[k] = 0.f;
        }
        // the copies of a short last tile share the columns
        int n = kRows, off = 0;
        const int short_qb = R.span < kRows ? n_qt - 1 : -1;
        const int n_short = R.span, off_short = (quarter * 32 / R.span) * R.span;
        bool on = false, any = false;
        int limit = 0;
        auto enter_tile = [&]() {
            on = (live >> qb) & 1u;
            any = __any_sync(0xffffffffu, on);
            n = qb == short_qb ? n_short : kRows;
            off = qb == short_qb ? off_short : 0;
            if (MASK) {
#pragma unroll
                for (int k = 0; k < kQTiles; ++k)
                    if (k == qb) limit = lim[k];
            }
        };
        enter_tile();
        while (t < t1) {
            if (!acquire()) return false;
            if (any) {
                const uint32_t ta = tmem + off;
                int nv = n;  // columns that hold keys
                if (t == cache_tiles - 1) nv = nv_cache - off;
                if (t == all_tiles - 1 && t >= cache_tiles) nv = nv_chunk - off;
                nv = min(nv, n);
                int nl = nv, full_cols = nv;
                if (MASK) {
                    nl = min(nv, limit - (t < cache_tiles ? t * kRows : u.c + (t - cache_tiles) * kRows) - off);
                    full_cols = __reduce_min_sync(0xffffffffu, on ? nl : nv);
                    nv = __reduce_max_sync(0xffffffffu, on ? nl : 0);
                }
                // a row's reference is the maximum of the first columns it meets
                if (nv > 0) {
                    if (__any_sync(0xffffffffu, st.m[0] == -INFINITY && on && nl > 0)) {
                        keep_branch();
                        uint32_t r[16];
                        tmem_ld_issue(ta, r);
                        tmem_ld_wait(r);
                        mask_tail(r, nl);
                        const float cmax = chunk_max(r);
                        if (st.m[0] == -INFINITY) st.m[0] = cmax;
                    }
                    uint64_t acc0 = 0, acc1 = 0;
                    const float negm = -(st.m[0] * scale2);
                    int cc = 0;
#pragma unroll 1
                    for (; cc + 32 <= full_cols; cc += 32) {
                        uint32_t r[32];
                        tmem_ld_issue(ta + cc, r);
                        tmem_ld_wait(r);
                        lse_sum<32>(r, scale2, negm, acc0, acc1);
                    }
                    const float zn = st.z[0] + sum_of(acc0, acc1);
                    if (__any_sync(0xffffffffu, !(zn <= 3.0e38f) && on && cc > 0)) {  // overflow: the whole visit, with care
                        keep_branch();
                        cc = 0;
                    } else if (cc > 0) {
                        st.z[0] = zn;
                    }
                    if (cc < nv) {
                        keep_branch();
                        const float2 s = lse_any<MASK>(ta + cc, n - cc, nv - cc, nl - cc, on, scale2, st.m[0], st.z[0]);
                        st.m[0] = s.x;
                        st.z[0] = s.y;
                    }
                }
            }
            release();
            if (n_qt != 3) {
                t += step;
            } else {
                keep_branch();
                ++t;
                if (++qb == 3) {
                    qb = 0;
                    ++t;
                }
                const float m0 = st.m[0], z0 = st.z[0];
                st.m[0] = st.m[1];
                st.z[0] = st.z[1];
                st.m[1] = st.m[2];
                st.z[1] = st.z[2];
                st.m[2] = m0;
                st.z[2] = z0;
                enter_tile();
            }
        }
        st.qb = qb;
        return true;
    }
    // This group's part of the rows' statistics; parts: [kGroups][stride] of the segment, from the chunk's first row on.
    __device__ __forceinline__ void store_stats(const Rows &R, const RowStats &s, uint32_t live, float2 *parts, int stride, bool nothing) const {
        float2 *dst = parts + (int64_t)s.rel * stride + my_row;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int qb = s.qb + k;
            if (qb >= R.n_qt) qb -= R.n_qt;
            if ((k == 0 || R.n_qt == 3) && ((live >> qb) & 1u)) dst[qb * kRows] = nothing ? make_float2(0.f, 0.f) : make_float2(s.m[k] * scale2, s.z[k]);
        }
    }
    // tail: columns at or beyond nv hold no row
    template <int NC, bool M>
    __device__ __forceinline__ void colsum_cols(uint32_t taddr, bool tail, int nv, uint32_t sm4, float &c0, float &c1, const int *lim, int j) {
        uint32_t r[NC];
        tmem_ld_issue(taddr, r);
        tmem_ld_wait(r);
        if (tail) mask_tail(r, nv);
        colsum_chunk<NC, M>(r, scale2, sm4, c0, c1, (const int2 *)lim, j);
    }
    // n columns (a multiple of 16) of one key tile against staged rows row ..: the key's column sum over nv of them.
    __device__ __forceinline__ float colsum_visit(uint32_t ta, int n, int nv, uint32_t sm4, const int *lim, const int2 *bounds,
                                                  int row, int j) {
        float c0 = 0.f, c1 = 0.f;
        bool all = true;  // every row sees every key of the warp
        const int j_lo = j - lane, j_hi = j_lo + 31;
        if (MASK) {
            const int2 lim16 = bounds[(row + min(lane & 7, (n >> 4) - 1) * 16) >> 4];
            if (j_lo >= __reduce_max_sync(0xffffffffu, lim16.y)) return 0.f;  // no row sees any of them
            all = j_hi < __reduce_min_sync(0xffffffffu, lim16.x);
        }
        int cc = 0;
        if (all) {
#pragma unroll 1
            for (; cc + 32 <= nv; cc += 32) colsum_cols<32, false>(ta + cc, false, 32, sm4 + cc * 8, c0, c1, nullptr, 0);
            if (cc < n) {
                keep_branch();
#pragma unroll 1
                for (; cc < n; cc += 16) colsum_cols<16, false>(ta + cc, true, nv - cc, sm4 + cc * 8, c0, c1, nullptr, 0);
            }
        } else {
            keep_branch();
#pragma unroll 1
            for (; cc < n; cc += 16) {
                const int2 b = bounds[(row + cc) >> 4];
                if (j_lo >= b.y) continue;  // no row of these sees any key of the warp
                if (j_hi < b.x)
                    colsum_cols<16, false>(ta + cc, nv - cc < 16, nv - cc, sm4 + cc * 8, c0, c1, nullptr, 0);
                else
                    colsum_cols<16, true>(ta + cc, nv - cc < 16, nv - cc, sm4 + cc * 8, c0, c1, lim + row + cc, j);
            }
        }
        return c0 + c1;
    }
    // Second sweep over key tiles [t0, t1) against the staged statistics `stats` (and limits): column sums to the writer, or,
    // DIRECT, for units of one query tile, whose keys have no other rows, to `scores`.
    template <bool DIRECT = false>
    __device__ __forceinline__ bool colsum_segment(const UnitInfo &u, const Rows &R, int t0, int t1, const float2 *stats,
                                                   const int *lim, const int2 *bounds, float *scores = nullptr) {
        const int n_st = R.n_st, kt = R.kt;
        const uint32_t first = (group - A) & 3, sm = smem_u32(stats);
        const uint32_t sum_full = smem_u32(c.sum_full), sum_empty = smem_u32(c.sum_empty);
        const int cols = (R.rows + 15) & ~15;
        int s = first % n_st, t = t0 + (first / n_st) * kt;
        const int step = n_st == 1 ? 4 * kt : (n_st == 2 ? 2 : 1);
        const uint32_t n_acc = kt == 2 ? (t1 - t0 + 1) >> 1 : (t1 - t0) * n_st, E0 = E;
        A += n_acc;
        E += n_acc;
        for (uint32_t a = E0 + first; t < t1; a += 4) {
            if (!acquire()) return false;
            const int row = s * R.width, n = min(R.width, cols - row), nv = min(n, R.rows - row);
            const uint32_t sm4 = sm + row * 8;
            const float v0 = colsum_visit(tmem, n, nv, sm4, lim, bounds, row, MASK ? key_tile(u, t).j0 + my_row : 0);
            float v1 = 0.f;
            if (kt == 2 && t + 1 < t1)
                v1 = colsum_visit(tmem + kRows / 2, n, nv, sm4, lim, bounds, row, MASK ? key_tile(u, t + 1).j0 + my_row : 0);
            release();
            if (DIRECT) {
                const KeyTile k0 = key_tile(u, t);
                if (my_row < k0.valid) scores[k0.j0 + my_row] = v0;
                if (kt == 2 && t + 1 < t1) {
                    const KeyTile k1 = key_tile(u, t + 1);
                    if (my_row < k1.valid) scores[k1.j0 + my_row] = v1;
                }
                t += step;
                continue;
            }
            const uint32_t buf = a % kSumBufs;
            if (!__all_sync(0xffffffffu, mbar_wait(sum_empty + buf * 8, ((a / kSumBufs) & 1) ^ 1, c.abort_flag))) return false;
            float *out = c.sums + buf * 2 * kRows + my_row;
            out[0] = v0;
            if (kt == 2) out[kRows] = v1;
            __syncwarp();
            if (lane == 0) mbar_arrive(sum_full + buf * 8);
            if (n_st != 3) {
                t += step;
            } else {
                ++t;
                if (++s == 3) {
                    s = 0;
                    ++t;
                }
            }
        }
        return true;
    }
};

// The parts of a row's statistics, numbered: per segment, copy of the row, and group that met its query tile.  A segment
// stores a group's part at the position of the group's first accumulator, so that with one, two or four query tiles the
// parts of tile qb are at positions qb, qb + n_qt, ...; with three at all four.  Accumulator a of a segment is query tile a % n_qt, so
// segments of one or two key tiles (`tiles`, at most) hold no more parts of a tile than that, at positions qb, qb + n_qt, ... modulo
// four: of three query tiles in ranges of one key tile one in four places is written (reading all of them from the cluster's
// shared memory took 11 us of a call of 28).
struct Parts {
    int log_p, log_c, first, step, span;
    __device__ Parts(const Rows &R, int qb, int tiles = kGroups) {
        const bool last = qb == R.n_qt - 1;
        log_c = !last || R.span == 128 ? 0 : (R.span == 64 ? 1 : 2);
        log_p = min(R.n_qt == 4 ? 0 : (R.n_qt == 2 ? 1 : 2), tiles == 1 ? 0 : (tiles == 2 ? 1 : 2));
        const bool all = R.n_qt == 3 && log_p == 2;
        first = all ? 0 : qb;
        step = all ? 1 : (R.n_qt < 3 ? R.n_qt : (qb == 0 ? 3 : -1));  // of three: qb and the position three on, modulo four
        span = R.span;
    }
    __device__ int count(int segments) const { return segments << (log_p + log_c); }
    __device__ int segment(int k) const { return k >> (log_p + log_c); }
    // offset of part k in [segments][kGroups][stride], from the row's own slot on
    __device__ int64_t at(int k, int stride) const {
        const int p = k & ((1 << log_p) - 1), c = (k >> log_p) & ((1 << log_c) - 1), s = k >> (log_p + log_c);
        return (int64_t)(s * kGroups + first + p * step) * stride + c * span;
    }
};

// ------------------------------------------------------------------------------------------------ column-sum writer
struct SumWriter {
    const Cta &c;
    int lane;
    uint32_t A = 0;  // accumulators of the second-sweep segments so far
    // Key tiles [t0, t1) of a second-sweep segment: the row blocks' sums of a key, added in block order, to
    // out[candidate]; `add`: a later row chunk of the same unit adds to what the earlier ones wrote (by this same warp).
    __device__ bool segment(const UnitInfo &u, const Rows &R, int t0, int t1, float *out, bool add) {
        for (int t = t0; t < t1; t += R.kt) {
            float v[2][kRows / 32];
#pragma unroll
            for (int i = 0; i < kRows / 32; ++i) v[0][i] = v[1][i] = 0.f;
            for (int s = 0; s < R.n_st; ++s, ++A) {
                const uint32_t buf = A % kSumBufs;
                const bool ok = mbar_wait_relaxed(&c.sum_full[buf], (A / kSumBufs) & 1, c.abort_flag, 500);
                if (!__all_sync(0xffffffffu, ok)) return false;
                const float *src = c.sums + buf * 2 * kRows + lane;
#pragma unroll
                for (int i = 0; i < kRows / 32; ++i) {
                    v[0][i] += src[i * 32];
                    if (R.kt == 2) v[1][i] += src[kRows + i * 32];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.sum_empty[buf]);
            }
            for (int k = 0; k < R.kt && t + k < t1; ++k) {
                const KeyTile kt = key_tile(u, t + k);
#pragma unroll
                for (int i = 0; i < kRows / 32; ++i) {
                    const int row = i * 32 + lane;
                    if (row < kt.valid) {
                        float *dst = out + kt.j0 + row;
                        const float x = k ? v[1][i] : v[0][i];
                        *dst = add ? *dst + x : x;
                    }
                }
            }
        }
        return true;
    }
    // Tiles of a request without prompt rows: the empty sum.
    __device__ void zeros(const UnitInfo &u, int t0, int t1, float *out) {
        for (int t = t0; t < t1; ++t) {
            const KeyTile kt = key_tile(u, t);
            for (int row = lane; row < kt.valid; row += 32) out[kt.j0 + row] = 0.f;
        }
    }
};

}  // namespace tc
}  // namespace finch
