// Prompt-guided scoring with both sweeps in ONE persistent kernel (single-request batches, bf16, head_dim 64/128,
// at most 512 padded query rows per KV head, or, in small calls, per half of its query heads; no per-row mask).
//
// The logits S = Q K^T of a unit (layer, KV head) are visited twice -- the row log-sum-exp must be known before any
// column sum can be formed -- but here the second visit follows the first closely enough that the keys come back
// from L2 instead of HBM, and nothing but a few bytes per prompt row leaves the SM in between:
//
//   * The key tiles of all units form one sequence (unit-major).  It is cut into ranges of W tiles, the last
//     of a unit possibly shorter; CTA i of the persistent grid takes ranges i, i + P, i + 2P, ... (one "window" each), so the
//     CTAs of a window work on neighbouring tiles and the keys in flight between the two sweeps of a window are P x W
//     tiles (tens of MB).
//   * Phase A of a window: D = Qtile x Ktile^T (one prompt row per TMEM lane), every softmax thread keeps the
//     (reference, sum exp2) of its rows over the window's tiles, publishes them to a small global array and bumps
//     the unit's ticket.  Nobody waits in phase A.
//   * Phase B: wait (bounded) until the ticket shows that every range of the unit has published -- the other
//     ranges belong to neighbouring CTAs that run phase A of the same window at the same time -- merge the parts
//     in a fixed order into (-R, w) per row, stage them in shared memory, then D = Ktile x Qrows^T (one key per
//     lane) and each thread sums exp2(s - R_r) w_r over a block of the prompt rows; the column-sum warp adds the
//     blocks of a key in order.
//   * With several windows per CTA phase A of window k + 1 runs before phase B of window k, so the tickets are long
//     complete when phase B needs them, and one warp does the merging meanwhile.  With a single window per CTA (a
//     layer at a time: the call is latency) all softmax warps merge at once.
//
// Tickets live in the context and are zero between calls (tickets.h).
#include "score_roles.cuh"
#include "tickets.h"

#include <climits>
#include <type_traits>

namespace finch {
namespace {

using namespace ptx;
using namespace tc;

constexpr int kMaxSegs = 64;  // ranges per unit (each prompt row merges a few statistics of every range)

struct FusedParams {
    ModelView mv;  // the scoring view: one unit per KV head, or two of half its query heads
    BatchView bv;
    float2 *partial;     // [units][n_seg][kGroups][rows_alloc] (reference base-2 logit, sum exp2) per row and part
    int *tickets;        // [2][units] the two counters of a unit
    float *row_lse;      // nullable
    float *unit_scores;  // [units][cand]: the column sums of a unit's query heads
    int *status;
    int W;           // key tiles per range
    int n_seg;       // ranges per unit, from the host bounds (the device's lengths may need fewer)
    int stages;      // key-tile ring depth
    int rows_alloc;  // query rows of a unit, whole tiles
    int q_tiles;     // query tiles the shared memory holds
    int cluster;     // CTAs of a cluster: the unit's ranges, with one window and few ranges per unit; else 1
    int key_shift;   // units that share a KV head, as a power of two (scoring_view)
};

__device__ __forceinline__ int ld_acquire_gpu(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Bounded wait for a global counter to reach `target` (about a second); gives up as soon as another thread of the
// CTA has, and then raises *abort_flag like the mbarrier waits.
constexpr uint32_t kTicketSpins = 1u << 21;
__device__ __forceinline__ bool ticket_wait(const int *ticket, int target, volatile int *abort_flag) {
    for (uint32_t it = 0; it < kTicketSpins; ++it) {
        if (ld_acquire_gpu(ticket) >= target) return true;
        if (*abort_flag) return false;
        if (it >= 8) __nanosleep(it < 256 ? 40 : 400);
    }
    *abort_flag = 1;
    return false;
}

// A counter in shared memory that the softmax warps bump (after their writes) and the statistics warp polls (before
// its reads): a plain counter, not a barrier phase, so that a reader that falls behind still reads the right answer.
__device__ __forceinline__ void count_arrive(int *counter) {
    __threadfence_block();
    atomicAdd_block(counter, 1);
}
__device__ __forceinline__ bool count_wait(int *counter, int target, volatile int *abort_flag) {
    for (uint32_t it = 0; it < kTicketSpins; ++it) {
        if (*(volatile int *)counter >= target) {
            __threadfence_block();
            return true;
        }
        if (*abort_flag) return false;
        __nanosleep(500);
    }
    *abort_flag = 1;
    return false;
}

struct Seg {
    int sweep, unit, t0, t1, slot, win;
};

// The segments of one CTA, in order: phase A of window k, then phase B of window k - delay (0 with one window, 1 with several).
struct Walk {
    int W, T, n_seg, delay, n_win, step, ph;
    __device__ bool next(Seg &s) {
        for (; step < n_win + delay; ph ? (ph = 0, ++step) : (ph = 1)) {
            const int win = step - (ph ? delay : 0);
            if (win < 0 || win >= n_win) continue;
            const int rho = win * (int)gridDim.x + (int)blockIdx.x;
            s.sweep = ph;
            s.win = win;
            s.unit = rho / n_seg;
            s.slot = rho - s.unit * n_seg;
            s.t0 = s.slot * W;
            s.t1 = max(s.t0, min(T, s.t0 + W));
            ph ? (ph = 0, ++step) : (ph = 1);
            return true;
        }
        return false;
    }
};

// (M, Z) of a prompt row -> what the second sweep needs, and the row's log-sum-exp where it is asked for.
__device__ __forceinline__ float2 finish_row(const FusedParams &p, const UnitInfo &u, const Rows &R, int row, float M, float Z,
                                             bool write_lse) {
    if (p.bv.self_lse || (write_lse && p.row_lse)) {
        const int64_t at = ((int64_t)u.l * p.mv.Hq + u.G * p.mv.hpg + row / R.rp) * p.bv.total_q + u.q0 + row % R.rp;
        if (p.bv.self_lse) merge_self_term(p.bv.self_lse[at], M, Z);
        if (write_lse && p.row_lse) p.row_lse[at] = merged_lse(M, Z);
    }
    return merged_pair(M, Z);
}

// The second sweep reads its rows in blocks of 16: the rows behind the last one of a unit are staged with weight 0.
__device__ __forceinline__ int staged_rows(const Rows &R) { return (R.rows + 15) & ~15; }

// The statistics of a unit, merged over its ranges and the parts of each range in a fixed order and staged, by one warp:
// four rows and four parts of each per lane in flight.
__device__ __forceinline__ void merge_by_warp(const FusedParams &p, const UnitInfo &u, const Rows &R, int n_seg, int unit,
                                              bool write_lse, float2 *stats, int lane) {
    const float2 *src = p.partial + (int64_t)unit * p.n_seg * kGroups * p.rows_alloc;
    for (int qb = 0; qb < R.n_qt; ++qb) {
        const Parts parts(R, qb);
        const int n = parts.count(n_seg), row0 = qb * kRows + lane;
        bool live[4];
        float M[4], Z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            live[k] = row_live(R, row0 + k * 32);
            M[k] = -INFINITY;
            Z[k] = 0.f;
        }
#pragma unroll 1
        for (int i0 = 0; i0 < n; i0 += 4) {
            float2 part[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 *at = src + parts.at(i0 + i, p.rows_alloc) + row0;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    part[k][i] = i0 + i < n && live[k] ? __ldcg(at + k * 32) : make_float2(0.f, 0.f);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) merge_parts(part[k], M[k], Z[k]);
        }
        int live_k = live[0] | live[1] << 1 | live[2] << 2 | live[3] << 3;
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const int row = row0 + k * 32;
            if (row < staged_rows(R))
                stage_row(stats, row, live_k & 1 ? finish_row(p, u, R, row, M[0], Z[0], write_lse) : make_float2(0.f, 0.f));
            live_k >>= 1;
            M[0] = M[1], M[1] = M[2], M[2] = M[3];
            Z[0] = Z[1], Z[1] = Z[2], Z[2] = Z[3];
        }
    }
}

// The same by all softmax threads: a row per thread, or, for few rows, per 2 to 16 neighbouring lanes that take every
// second to sixteenth part each (many short ranges leave hundreds of parts to a row).  `remote`: shared-memory address of
// the parts, the same in every CTA of the cluster, or 0: they are in global memory.  What a part's address costs counts: a row of a
// short last tile has four parts to a range (4 units of 31 ranges x 400 rows 30.2 us with a condition on each load and the
// positions taken modulo four in it, 26.0 so).
__device__ __forceinline__ void merge_by_cta(const FusedParams &p, const UnitInfo &u, const Rows &R, int n_seg, int unit,
                                             bool write_lse, float2 *stats, int tid, uint32_t remote) {
    const float2 *src = p.partial + (int64_t)unit * p.n_seg * kGroups * p.rows_alloc;
    int log_s = 0;  // lanes per row
    while (log_s < 4 && R.rows << (log_s + 1) <= kSoftmaxWarps * 32) ++log_s;
    const int row = tid >> log_s, sub = tid & ((1 << log_s) - 1);
    const bool live = row_live(R, row);
    const Parts parts(R, live ? row / kRows : 0, p.W);
    const int n = live ? parts.count(n_seg) : 0;
    float M = -INFINITY, Z = 0.f;
#pragma unroll 1
    for (int i0 = sub; i0 < n; i0 += 8 << log_s) {
        float2 part[8];
        if (remote) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int k = i0 + (i << log_s), seg = parts.segment(k);
                const uint32_t at = (uint32_t)parts.at(k - (seg << (parts.log_p + parts.log_c)), p.rows_alloc) + row;
                part[i] = k < n ? ld_remote(map_to_rank(remote + at * 8, seg)) : make_float2(0.f, 0.f);
            }
        } else {
            // (loads without a condition: eight in flight; a lane with fewer parts left reads its last one again)
#pragma unroll
            for (int i = 0; i < 8; ++i) part[i] = __ldcg(src + parts.at(min(i0 + (i << log_s), n - 1), p.rows_alloc) + row);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i0 + (i << log_s) >= n) part[i] = make_float2(0.f, 0.f);
        }
        merge_parts(part, M, Z);
    }
    for (int d = 1; d < 1 << log_s; d <<= 1) {  // only the first lane's value is used
        const float om = __shfl_xor_sync(0xffffffffu, M, d), oz = __shfl_xor_sync(0xffffffffu, Z, d);
        const float nm = fmaxf(M, om);
        if (nm != -INFINITY) Z = Z * ex2(M - nm) + oz * ex2(om - nm);
        M = nm;
    }
    if (sub == 0 && row < staged_rows(R))
        stage_row(stats, row, live ? finish_row(p, u, R, row, M, Z, write_lse) : make_float2(0.f, 0.f));
}

// One window: the first softmax thread signs off for the CTA's range when its warp gives up.
__device__ __noinline__ void give_up(int *published, int *left, int ranges, int unit, bool publish) {
    if (threadIdx.x != kCtlWarps * 32) return;
    const Tickets tickets{published, left, ranges};
    if (publish) tickets.publish(unit);
    tickets.leave(unit);
}

// PAIR: units of one query tile, and no column sums to be added: the writer's warp is a second MMA issuer, the softmax warps write.
// ONE: a CTA has one window at most, and the softmax warps merge the statistics themselves.  (Kernels of their own: with either merge
// in the other's kernel its loops came out by up to 2 % slower or faster as the other's code changed.  32 x 32 units of 8 key tiles x
// 64 rows 89.3 -> 87.6 us, 32 x 8 of 27 x 256 165.0 -> 160.6, 28 x 8 of 9 x 160 52.6 -> 51.4, 192 of 8 x 64, head_dim 64, 24.2 -> 23.1.)
template <int D, bool PAIR, bool ONE>
__global__ void __launch_bounds__(kTcThreads, 1)
score_fused_kernel(const __grid_constant__ CUtensorMap q_big, const __grid_constant__ CUtensorMap q_small,
                   const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap chunk_map,
                   FusedParams p) {
    extern __shared__ uint8_t smem_raw[];
    const Cta c = cta_layout(smem_raw, (D / 64) * kSlabBytes, p.q_tiles, p.rows_alloc, p.stages);
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp-uniform for the compiler
    const int cluster = ONE ? p.cluster : 1;
    if (threadIdx.x == 0) {
        prefetch_tensormap(&q_big);
        prefetch_tensormap(&q_small);
        prefetch_tensormap(&cache_map);
        prefetch_tensormap(&chunk_map);
    }
    const uint32_t tmem = cta_setup(c, ONE ? kSoftmaxWarps : 1, cluster, PAIR ? 2 : 1);
    // The inputs were written by what precedes this kernel.  The successor is NOT allowed to launch early: its CTAs
    // would take over the SMs of the CTAs that finish first and park there in their wait (measured: + 20 us on the
    // 0.5 ms step of 32 layers x 8 KV heads x 4096 candidates).
    dependency_wait();

    UnitInfo u = unit_info(mv, bv, 0, 0);  // l and G are set per segment
    const Rows R = make_rows(u.n_q, mv.hpg, 0);
    const int T = n_key_tiles(u), n_seg = cluster > 1 ? p.n_seg : (T + p.W - 1) / p.W;
    const bool run = u.ok && u.n_q > 0 && u.N > 0;
    const int n_ranges = mv.L * mv.G * n_seg;
    const int n_win = run && (int)blockIdx.x < n_ranges ? (n_ranges - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    if (!u.ok && threadIdx.x == 0 && blockIdx.x == 0) atomicOr(p.status, FINCH_DEV_BAD_BATCH);
    const Tickets tickets{p.tickets, p.tickets + mv.L * mv.G, n_seg};
    Walk walk{p.W, T, n_seg, ONE ? 0 : 1, n_win, 0, 0};
    Seg sg;
    bool ok = true, left = false;
    // With several windows the sweeps of two units alternate.  Where the ring holds both their query tiles a window loads
    // its queries once and keeps them for its second sweep (64 rows: 0.105 -> 0.09 ms for 1024 units of 8 key tiles).
    const bool retain = !ONE && 2 * R.n_qt <= p.q_tiles;
    TileRing ring{p.q_tiles};
#define FINCH_UNIT(s) (u.l = (s).unit / mv.G, u.G = (s).unit % mv.G)

    if (warp == 0) {
        Producer<D, false, true> role{c, &q_big, &q_small, &cache_map, &chunk_map, mv.hpg, bv.total_q, p.key_shift};
        int q_unit = -1;
        while (ok && walk.next(sg)) {
            FINCH_UNIT(sg);
            const bool reload = retain ? sg.sweep == 0 : q_unit != sg.unit;
            q_unit = sg.unit;
            if (sg.t0 < sg.t1) ok = role.segment(u, R, sg.t0, sg.t1, reload ? ring.take(R.n_qt) : -1);
        }
        role.drain();
    } else if (warp == 1 || (PAIR && warp == 3 && u.n_q > 0)) {
        Issuer<D, PAIR> role(c, tmem, warp >> 1);
        int q_unit = -1, odd = 0, even = 0;  // query tiles of the odd and the even windows
        Seg nx;
        for (bool more = walk.next(sg); ok && more; sg = nx) {
            more = walk.next(nx);
            if (sg.t0 >= sg.t1) continue;  // a cluster's CTA beyond the unit's last tile
            const bool reload = retain ? sg.sweep == 0 : q_unit != sg.unit;
            const bool release = retain ? sg.sweep == 1 : more && nx.unit != sg.unit;
            q_unit = sg.unit;
            if (reload) {
                const int at = ring.take(R.n_qt);
                if (!retain || (sg.win & 1)) odd = at;
                if (!retain || !(sg.win & 1)) even = at;
            }
            const int base = sg.win & 1 ? odd : even;
            ok = sg.sweep == 0 ? role.lse_segment(R, sg.t0, sg.t1, base, reload, release)
                               : role.colsum_segment(R, sg.t0, sg.t1, base, reload, release);
        }
    } else if (warp == 2) {
        // statistics warp: makes a phase-A segment's statistics visible to the GPU, bumps the unit's ticket, waits until
        // every range of the unit has published and stages the merged rows for the segment's phase B, which the softmax
        // warps reach one phase A later.  Two buffers in turn: this warp cannot be two segments ahead, it waits for
        // the softmax warps' phase A in between.
        if (!ONE) {
            int segs = 0, good = 1;
            while (walk.next(sg)) {
                if (sg.sweep) continue;
                ++segs;
                FINCH_UNIT(sg);
                if (lane == 0)  // a range that gives up still signs off, and so do those behind it
                    good = tickets.pass(
                        sg.unit, good,
                        [&]() {
                            const bool written = count_wait(c.a_count, kSoftmaxWarps * segs, c.abort_flag);
                            __threadfence();  // cumulative: covers the softmax warps' stores this thread has synchronised with
                            return written;
                        },
                        [&](const int *ticket, int n) { return ticket_wait(ticket, n, c.abort_flag); });
                if (!__shfl_sync(0xffffffffu, good, 0)) continue;
                merge_by_warp(p, u, R, n_seg, sg.unit, sg.slot == 0, c.stats + ((segs - 1) & 1) * p.rows_alloc, lane);
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.stats_ready[(segs - 1) & 1]);
            }
        }
    } else if (warp == 3) {
        SumWriter role{c, lane};
        const int64_t cand = (int64_t)bv.total_cache + bv.total_chunk;
        if (u.ok && u.n_q == 0)  // no prompt rows: the empty sum
            for (int unit = blockIdx.x; unit < mv.L * mv.G; unit += gridDim.x)
                role.zeros(u, 0, T, p.unit_scores + unit * cand + u.cache0 + u.chunk0);
        while (ok && walk.next(sg)) {
            if (!sg.sweep) continue;
            ok = role.segment(u, R, sg.t0, sg.t1, p.unit_scores + sg.unit * cand + u.cache0 + u.chunk0, false);
        }
    } else {
        Softmax<false> role(c, tmem, mv.scale * kLog2e);
        uint32_t live = 0;  // bit qb: this thread's row of query tile qb is a prompt row
#pragma unroll
        for (int qb = 0; qb < kQTiles; ++qb)
            if (qb < R.n_qt && row_live(R, role.row_of(R, qb))) live |= 1u << qb;
        const int no_limit[kQTiles] = {};
        int segs_b = 0;
        while (ok && walk.next(sg)) {
            if (sg.sweep == 0) {
                Softmax<false>::RowStats st;
                if (!(ok = role.lse_segment(u, R, sg.t0, sg.t1, live, no_limit, st))) {
                    if (ONE && cluster == 1) give_up(tickets.published, tickets.left, n_seg, sg.unit, true);
                    break;
                }
                if (cluster > 1) {
                    // the unit's ranges are the CTAs of this cluster: the parts stay in shared memory, every warp tells
                    // every CTA that its own are written
                    float2 *parts = c.stats + 2 * p.rows_alloc;
                    role.store_stats(R, st, live, parts, p.rows_alloc, false);
                    __syncwarp();
                    cluster_wait();  // everybody's barriers are initialised
                    if (lane < cluster) mbar_arrive_remote(map_to_rank(smem_u32(c.parts_ready), lane));
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait_cluster(c.parts_ready, 0, c.abort_flag)))) {
                        cluster_arrive();
                        left = true;
                        break;
                    }
                    FINCH_UNIT(sg);
                    merge_by_cta(p, u, R, n_seg, sg.unit, sg.slot == 0, c.stats, threadIdx.x - kCtlWarps * 32, smem_u32(parts));
                    __syncwarp();
                    cluster_arrive();  // through with the neighbours' shared memory
                    left = true;
                    if (lane == 0) mbar_arrive(&c.stats_ready[1]);
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&c.stats_ready[1], 0, c.abort_flag)))) break;
                    continue;
                }
                role.store_stats(R, st, live, p.partial + ((int64_t)sg.unit * p.n_seg + sg.slot) * kGroups * p.rows_alloc, p.rows_alloc,
                                 false);
                __syncwarp();
                if (!ONE) {
                    if (lane == 0) count_arrive(c.a_count);
                    continue;
                }
                // one window: publish, wait for the other ranges of the unit, merge a row per thread
                const int tid = threadIdx.x - kCtlWarps * 32;
                if (lane == 0) mbar_arrive(&c.stats_ready[0]);
                int good = 1;
                if (lane == 0) {
                    if (tid == 0) {
                        good = mbar_wait(&c.stats_ready[0], 0, c.abort_flag);
                        __threadfence();  // cumulative, as above
                        tickets.publish(sg.unit);
                    }
                    good = good && ticket_wait(&p.tickets[sg.unit], n_seg, c.abort_flag);
                }
                if (!(ok = __shfl_sync(0xffffffffu, good, 0))) {
                    give_up(tickets.published, tickets.left, n_seg, sg.unit, false);
                    break;
                }
                FINCH_UNIT(sg);
                merge_by_cta(p, u, R, n_seg, sg.unit, sg.slot == 0, c.stats, tid, 0);
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.stats_ready[1]);
                ok = __all_sync(0xffffffffu, mbar_wait(&c.stats_ready[1], 0, c.abort_flag));
                if (tid == 0) tickets.leave(sg.unit);  // every warp of this CTA has seen the ticket complete, or gives up
                if (!ok) break;
            } else {
                const int b = ONE ? 0 : segs_b & 1;
                if (!ONE && !(ok = __all_sync(0xffffffffu, mbar_wait(&c.stats_ready[b], (segs_b >> 1) & 1, c.abort_flag)))) break;
                ok = role.template colsum_segment<PAIR>(u, R, sg.t0, sg.t1, c.stats + b * p.rows_alloc, nullptr, nullptr,
                                                        p.unit_scores + sg.unit * ((int64_t)bv.total_cache + bv.total_chunk) + u.cache0 + u.chunk0);
                ++segs_b;
            }
        }
    }
#undef FINCH_UNIT
    cta_teardown(c, tmem, p.status, cluster, left);
}

// scores of a selection group that spans several KV heads (one group per layer): the heads' column sums, added in
// head order.
__global__ void __launch_bounds__(256)
sum_heads_kernel(ModelView mv, BatchView bv, const float *unit_scores, float *scores, int out_groups, int heads_per_group) {
    dependency_wait();
    const int64_t cand = (int64_t)bv.total_cache + bv.total_chunk;
    const int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const int l = blockIdx.y / out_groups, og = blockIdx.y % out_groups;
    const UnitInfo u = unit_info(mv, bv, 0, blockIdx.z);
    if (!u.ok || j >= u.N) return;
    const int64_t at = (int64_t)u.cache0 + u.chunk0 + j;
    float s = 0.f;
    for (int k = 0; k < heads_per_group; ++k) s += unit_scores[((int64_t)l * mv.G + og * heads_per_group + k) * cand + at];
    scores[((int64_t)l * out_groups + og) * cand + at] = s;
}

// Key tiles per range, or 0 when the one-kernel path should leave the batch to the two-launch kernels.
//
// The estimate is in units of one query tile against one key tile in both sweeps, 2500 SM clocks where the pipeline is full:
//   one range per CTA        W x query tiles (0.7 W for at most 64 rows) + 4, + 0.3 for every eight parts of a row that a lane of
//                            the merge reads (merge_rounds): nothing hides the query load and the exchange of the row statistics.
//                            As a cluster, where all units' clusters run at once, the ranges of a unit exchange for 1 at 16 of
//                            them; else for 1.5 and, as the CTAs that poll, up to 1 more; + 0.5 for single tiles (36 units of
//                            8 key tiles x 96 rows: 17.2 us in ranges of 2 tiles, whose 36 clusters of 4 do not fit, 13.4 in
//                            ranges of 3; 2 units of 27 x 256 14.5 us in 27 ranges without a cluster, 18.5 in clusters of 14);
//   several ("windows")      windows x (W x query tiles + 2), or + 5 where the ranges of a unit meet across CTAs and are too
//                            short to hide it (28 x 8 units of 9 key tiles x 160 rows: whole units 55 us although a quarter
//                            of the second window's CTAs idle, ranges of 3 tiles 82 us);
//   two launches             the work spread evenly with 1.2 of the time per accumulator, + 14 for launches and merge; against several
//                            windows + 10 and 1.7 per accumulator where a key tile has only one or two (77 us in the example).
// The constants are fits to 1450 calls of 1 to 1300 units, 2 to 32 key tiles and 8 to 512 rows, where the chosen way takes 1.009 times
// as long as the best one in the geometric mean (1.022 with 5, 0.03 a part, 3 for any missing cluster and 10 for two launches, which
// sent few units with many short ranges to two launches: 2 units of 23 tiles x 24 rows 25.6 us, 12.8 in ranges of 2).
// halves: a unit is half the query heads of a KV head.  Both halves fetch the keys: several windows have to be better by a tenth, and
// are whole units, unless a divisor would be estimated better still: there two launches are shorter (24 x 32 units of 14 key tiles x
// 288 rows 564 us, 601 in whole units), as they are for units of fewer than twelve accumulators (176 of 2 x 320 rows 31.3 us, 35.7;
// 192 of 2 x 464 41.8, 44.5).
// With one range per CTA a unit's last range may be shorter.  Several windows: ranges that divide the unit, of at least four
// tiles (or the unit), at most 8 to a unit, and keys in flight between a window's sweeps that mostly stay in L2.
constexpr int kMaxCluster = 16;
// Clusters of so many CTAs, one to an SM, that a device of this kind says it holds.  An estimate, so that a plan needs no device: a
// launch asks (fits_clusters), and on a device that holds others the rule only loses time.
constexpr int kClusters[kMaxCluster + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7};
// Rounds of eight loads that a lane of merge_by_cta makes for a row of the last query tile, the one with copies, as Parts counts them.
int merge_rounds(int rows, int n_seg, int W) {
    const int q_tiles = (rows + kRows - 1) / kRows, last = rows - (q_tiles - 1) * kRows;
    const int met = W < 3 ? W : kGroups, groups = q_tiles == 4 ? 1 : (q_tiles == 2 ? min(2, met) : met);
    int lanes = 1;
    while (lanes < 16 && rows * lanes * 2 <= kSoftmaxWarps * 32) lanes *= 2;
    return (n_seg * groups * (last <= 32 ? 4 : (last <= 64 ? 2 : 1)) + 8 * lanes - 1) / (8 * lanes);
}
int choose_window(long long units, int T, int ctas, int tile_bytes, int rows, bool halves) {
    const int q_tiles = (rows + kRows - 1) / kRows;
    const long long l2_budget = 120ll << 20;
    int best = 0;
    // in tenths: two launches as the limit of several windows and of one, a key tile of units of at most 64 rows
    const long long all = units * T * q_tiles, two_launches = all * (q_tiles <= 2 ? 17 : 12) / ctas + 100, two_small = all * 12 / ctas + 140;
    const int tile = rows <= kRows / 2 ? 7 : q_tiles * 10;
    long long best_cost = LLONG_MAX, barred = LLONG_MAX;
    bool several = false;
    for (int W = 1; W <= T; ++W) {
        const int n_seg = (T + W - 1) / W;
        if (n_seg > kMaxSegs || (W > 1 && n_seg == (T + W - 2) / (W - 1))) continue;  // longer, but no fewer ranges
        const long long ranges = units * n_seg, windows = (ranges + ctas - 1) / ctas;
        long long cost;
        if (windows == 1) {
            const bool clusters = n_seg <= kMaxCluster && units <= kClusters[n_seg];
            cost = (long long)W * tile + 40 + 3 * merge_rounds(rows, n_seg, W);
            if (n_seg > 1) cost += (clusters ? n_seg * 10 / 16 : 15 + ranges * 10 / ctas) + (W == 1 ? 5 : 0);
        } else {
            if ((W < 4 && W < T) || n_seg > 8 || T % W || (long long)W * ctas * tile_bytes > l2_budget) continue;
            cost = windows * (W * q_tiles * 10 + (n_seg > 1 && W * q_tiles < 16 ? 50 : 20)) * (halves ? 11 : 10) / 10;
            if (halves && W < T) barred = min(barred, cost);
            if (halves && (W < T || W * q_tiles < 12)) continue;
        }
        if (cost < (windows == 1 ? two_small : two_launches) && cost < best_cost) {
            best_cost = cost;
            best = W;
            several = windows > 1;
        }
    }
    return several && barred <= best_cost ? 0 : best;
}

// The scoring view: a query head only ever meets its own KV head's keys, so a unit is a KV head.  One of more query rows than stay
// resident is two units of half its query heads each, where that suffices; their column sums are added afterwards, as those of
// a selection group's KV heads are.
ModelView scoring_view(const ModelView &model, const BatchView &bv) {
    ModelView mv = model;
    const int halves = padded_rows(bv.max_q, model.g) > kMaxRows && model.g % 2 == 0 ? 2 : 1;
    mv.G = mv.Hkv * halves;
    mv.hpg = mv.g / halves;
    mv.kvpg = 1;
    return mv;
}
int rows_alloc_of(const ModelView &mv, const BatchView &bv) {  // resident query rows: whole tiles (mv: the scoring view)
    return (padded_rows(bv.max_q, mv.hpg) + kRows - 1) / kRows * kRows;
}

// With one window the ranges of a unit may form a cluster and exchange their row statistics through each other's shared
// memory, where all units' clusters run at once (a cluster lies within one group of SMs, so fewer may fit than SMs would
// allow).  The exchange through global memory and tickets costs 5.7 us of a 16 us call: stores, fence, atomic, poll, loads.
template <int D, bool PAIR>
bool fits_clusters(const Ctx &ctx, int size, int units) {
    int16_t &known = ctx.clusters[(D == 128) + 2 * PAIR][size];  // clusters of this size at a time, + 1; 0: not asked yet
    int16_t now = known;
    if (now == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(size);
        cfg.blockDim = dim3(kTcThreads);
        cfg.dynamicSmemBytes = kSmemLimit;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = size;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, score_fused_kernel<D, PAIR, true>, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        now = (int16_t)(n + 1);
        if (ctx.on_own_device()) known = now;
    }
    return now > units;
}

template <int D, bool PAIR>
cudaError_t launch_fused_d(const Ctx &ctx, const CUtensorMap &qb, const CUtensorMap &qs, const CUtensorMap &cm,
                           const CUtensorMap &hm, FusedParams p, int n_ranges, int out_groups, int heads_per_group, float *scores,
                           cudaStream_t stream) {
    constexpr int kTileBytes = (D / 64) * kSlabBytes;
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    const int sms = ctx.sm_count > 0 ? ctx.sm_count : 148, n_qt = p.rows_alloc / kRows;
    const bool one = n_ranges <= sms;
    // room for the queries of the two units that alternate, and of a third that is being loaded where they are short
    p.q_tiles = one || n_qt > 2 ? n_qt : n_qt + 2;
    const auto kernel = one ? score_fused_kernel<D, PAIR, true> : score_fused_kernel<D, PAIR, false>;
    const int bit = kSmemFused + (D == 128) + 2 * PAIR + 4 * one;
    cudaError_t e = cudaSuccess;
    if (!ctx.smem_ready(bit)) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e == cudaSuccess && one) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        ctx.smem_set(bit);
    }
    p.cluster = one && p.n_seg > 1 && p.n_seg <= kMaxCluster && fits_clusters<D, PAIR>(ctx, p.n_seg, mv.L * mv.G) ? p.n_seg : 1;
    const int parts = p.cluster > 1 ? kGroups * p.rows_alloc * 8 : 0;  // the cluster's exchange of row statistics
    p.stages = kMaxStages;
    while (p.stages > 2 && cta_smem(kTileBytes, p.q_tiles, p.rows_alloc, p.stages, false) + parts > kSmemLimit) --p.stages;
    const int smem = cta_smem(kTileBytes, p.q_tiles, p.rows_alloc, p.stages, false) + parts;
    dim3 grid(n_ranges < sms ? n_ranges : sms);  // persistent and resident at once: phase B waits for neighbours
    e = launch_chained_cluster(kernel, p.cluster, grid, dim3(kTcThreads), smem, stream, qb, qs, cm, hm, p);
    ctx.launches += 1;
    if (e != cudaSuccess || heads_per_group == 1) return e;
    return launch_sum_heads(ctx, mv, bv, p.unit_scores, scores, out_groups, heads_per_group, stream);
}

}  // namespace

cudaError_t launch_sum_heads(const Ctx &ctx, const ModelView &mv, const BatchView &bv, const float *unit_scores, float *scores,
                             int out_groups, int heads_per_group, cudaStream_t stream) {
    dim3 grid((bv.max_cache + bv.max_chunk + 255) / 256, mv.L * out_groups, bv.batch);
    ctx.launches += 1;
    return launch_chained(sum_heads_kernel, grid, dim3(256), 0, stream, mv, bv, unit_scores, scores, out_groups, heads_per_group);
}

// Key tiles per window the fused kernel would use for this batch; 0: the batch is not one it takes (several
// requests, causal rows, more query rows per KV head than stay resident, no window length that fits: see choose_window).
int score_fused_window(const Ctx &ctx, const BatchView &bv) {
    if (!score_tc_supported(ctx) || bv.batch != 1 || bv.row_limit || bv.max_q == 0 || bv.max_cache + bv.max_chunk == 0)
        return 0;
    const ModelView mv = scoring_view(ctx.model, bv);
    const int rows = padded_rows(bv.max_q, mv.hpg), sms = ctx.sm_count > 0 ? ctx.sm_count : 148;
    if (rows > kMaxRows) return 0;
    const int tiles = (bv.max_cache + kRows - 1) / kRows + (bv.max_chunk + kRows - 1) / kRows;
    // Halves of a KV head's queries: with one window, where the calls are latency and two launches of two chunks of rows each take longer
    // (36 single requests of 1 to 12 layers, 129 to 256 prompt rows x 4 heads: scoring 1.3 times as fast, 1.45 the 27 that the rule
    // takes; 6 x 2 units of 9 key tiles x 992 rows 41.2 -> 25.0 us, 3 x 8 of 19 x 752 56.4 -> 46.5), and as whole units in several
    // (224 halves of 4 x 320 rows 51.4 -> 47.2, 256 of 10 x 384 105 -> 91, 1280 of 11 x 368 453 -> 408).  In shorter ranges of several
    // windows, whose statistics meet across CTAs, 11 x 8 units of 20 x 800 took 166 us instead of 146.  Where the estimates are within
    // 10 %, two launches (31 x 8 units of 17 x 832 325 us, 334 in halves; 24 x 8 of 12 x 576 136, 140), although some would be shorter
    // (14 x 8 of 8 x 896 100.6, 89.4).
    return choose_window((long long)mv.L * mv.G, tiles, sms, (mv.d / 64) * kSlabBytes, rows, mv.G != mv.Hkv);
}

namespace {
size_t scratch_of(const ModelView &model, const BatchView &bv, int n_seg) {
    const ModelView mv = scoring_view(model, bv);
    const size_t units = (size_t)mv.L * mv.G, cand = (size_t)bv.total_cache + bv.total_chunk;
    size_t n = units * n_seg * kGroups * rows_alloc_of(mv, bv);  // partial row statistics
    if (mv.G != model.G) n += (units * cand + 1) / 2;  // sums of the units of a selection group that spans several
    return n;
}
int tiles_of(const BatchView &bv) { return (bv.max_cache + kRows - 1) / kRows + (bv.max_chunk + kRows - 1) / kRows; }
}  // namespace

// The most that any batch within these bounds needs: a unit has at most as many ranges as give every SM one (one window),
// or eight.
size_t score_fused_scratch_bound(const Ctx &ctx, const BatchView &bv) {
    if (!score_tc_supported(ctx) || bv.batch == 0 || bv.max_q == 0) return 0;
    BatchView one = bv;
    while (one.max_q > 0 && padded_rows(one.max_q, ctx.model.g) > kMaxRows) one.max_q -= kRowPad;  // the longest prompt it takes
    const int sms = ctx.sm_count > 0 ? ctx.sm_count : 148, per_sm = sms / (ctx.model.L * ctx.model.Hkv);
    const int ranges = per_sm < 8 ? 8 : (per_sm < kMaxSegs ? per_sm : kMaxSegs), tiles = tiles_of(bv);
    const size_t whole = one.max_q > 0 ? scratch_of(ctx.model, one, tiles < ranges ? tiles : ranges) : 0;
    // halves of a KV head's queries, also where all its heads are too many for the shortest prompt: one range to an SM, or to a
    // unit, as many rows as stay resident, sums of every unit
    if (ctx.model.g % 2 || padded_rows(bv.max_q, ctx.model.g) <= kMaxRows || padded_rows(1, ctx.model.g / 2) > kMaxRows) return whole;
    const size_t units = 2 * (size_t)ctx.model.L * ctx.model.Hkv;
    const size_t half = (units > (size_t)sms ? units : sms) * kGroups * kMaxRows + (units * ((size_t)bv.total_cache + bv.total_chunk) + 1) / 2;
    return half > whole ? half : whole;
}

// Float2 entries of scratch the fused kernel needs for this batch (0: the batch is not one it takes).
size_t score_fused_scratch(const Ctx &ctx, const BatchView &bv) {
    const int W = score_fused_window(ctx, bv);
    return W ? scratch_of(ctx.model, bv, (tiles_of(bv) + W - 1) / W) : 0;
}

// Returns cudaErrorNotSupported (and launches nothing) when the batch is not one the fused kernel takes, the
// scratch is too small or the tensors cannot be described to the TMA unit.
cudaError_t launch_score_fused(const Ctx &ctx, const TensorView &q, const TensorView &cache_k, const TensorView &chunk_k,
                               const BatchView &bv, float *scores, float2 *scratch, size_t scratch_capacity,
                               float *row_lse, cudaStream_t stream) {
    const int W = score_fused_window(ctx, bv);
    if (W == 0 || scratch_capacity < scratch_of(ctx.model, bv, (tiles_of(bv) + W - 1) / W)) return cudaErrorNotSupported;
    const ModelView mv = scoring_view(ctx.model, bv);
    CUtensorMap qb, qs, cm, hm;
    if (!make_map(&qb, q, mv.d, bv.total_q, mv.Hq, mv.L, kBigBox)) return cudaErrorNotSupported;
    if (!make_map(&qs, q, mv.d, bv.total_q, mv.Hq, mv.L, kRowPad)) return cudaErrorNotSupported;
    const bool have_cache = bv.max_cache > 0, have_chunk = bv.max_chunk > 0;
    if (have_cache && !make_map(&cm, cache_k, mv.d, bv.total_cache, mv.Hkv, mv.L, kRows)) return cudaErrorNotSupported;
    if (have_chunk && !make_map(&hm, chunk_k, mv.d, bv.total_chunk, mv.Hkv, mv.L, kRows)) return cudaErrorNotSupported;
    if (!have_cache) cm = hm;  // never dereferenced: the request has no cache tiles
    if (!have_chunk) hm = cm;
    const int tiles = tiles_of(bv);
    const int units = mv.L * mv.G;
    FusedParams p{};
    p.mv = mv;
    p.bv = bv;
    p.W = W;
    p.n_seg = (tiles + p.W - 1) / p.W;
    p.rows_alloc = rows_alloc_of(mv, bv);
    p.partial = scratch;
    p.tickets = ctx.tickets;
    p.key_shift = mv.G == mv.Hkv ? 0 : 1;
    p.unit_scores = ctx.model.G == mv.G ? scores : (float *)(scratch + (size_t)units * p.n_seg * kGroups * p.rows_alloc);
    p.row_lse = row_lse;
    p.status = ctx.d_status;
    const int n_ranges = units * p.n_seg;
    const auto launch = [&](auto d, auto pair) {
        return launch_fused_d<decltype(d)::value, decltype(pair)::value>(ctx, qb, qs, cm, hm, p, n_ranges, ctx.model.G, mv.G / ctx.model.G,
                                                                         scores, stream);
    };
    const auto by_dim = [&](auto pair) {
        return mv.d == 64 ? launch(std::integral_constant<int, 64>(), pair) : launch(std::integral_constant<int, 128>(), pair);
    };
    return p.rows_alloc == kRows ? by_dim(std::true_type()) : by_dim(std::false_type());
}

}  // namespace finch
