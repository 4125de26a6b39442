// Prompt-guided scoring on the 5th-generation tensor cores in two launches (bf16 inputs, head_dim 64 or 128): ragged
// batches, causal query rows, prompts of more than 512 padded rows per KV head, tile counts the one-kernel path has no
// window for.
//
// One kernel template, two sweeps over the logits S = Q K^T of a unit (layer, KV head, request), built from the roles
// in score_roles.cuh.  A CTA owns a contiguous range of work items (item = one key split of one unit); the unit's query
// rows are resident, 512 at a time, while the key tiles of the split stream past them.
//
//   kLse     D = Qtile x Ktile^T lands in tensor memory with one prompt row per lane, so each thread keeps the
//            online (reference, sum exp2) of its own rows without cross-lane traffic -> partial row statistics.
//   kColsum  D = Ktile x Qrows^T: one key per lane, so the sum over prompt rows of exp2(s - R) w is a private
//            running sum per thread -> scores.
// merge_stats_kernel merges the partial statistics in between, in a fixed order.
#include "score_roles.cuh"

namespace finch {
namespace {

using namespace ptx;
using namespace tc;

enum { kLse = 0, kColsum = 1 };

struct TcParams {
    ModelView mv;
    BatchView bv;
    float2 *partial;   // [requests x units][splits][kGroups][slots] (reference base-2 logit, sum exp2) per row and part
    float2 *merged;    // [L][Hq][total_q] (-reference, weight) per prompt row after merging the parts
    float *row_lse;    // nullable
    float *unit_scores;  // [L][Hkv][total_cand]
    int *status;
    int splits;        // key splits per unit
    int slots;         // padded query rows per unit (host bound), whole tiles
    int stages;        // key-tile ring depth that fits beside the resident queries
    int rows_alloc;    // query rows worked on at a time, whole tiles
    int q_tiles;       // query tiles the shared memory holds
    int n_items;       // work items = splits x units x requests, walked by a persistent grid
    const int *bounds;              // [grid + 1] first item of every CTA (work-weighted), or null: equal item counts
    unsigned long long *work_prefix;  // [batch + 1] work of all items of the requests before b (plan scratch)
    // `mv` is the scoring view: one scoring unit per KV head
};

// One stop of a CTA's walk: a chunk of the unit's query rows against the consecutive key splits that the CTA holds of it
// (one load of the queries for all of them).
struct Stop {
    UnitInfo u;
    Rows R;
    int t0, t1;
    int split, n_splits, chunk;
    int64_t key;    // (unit, request)
    int64_t q_key;  // equal keys share their query tiles
};

// A role's position in its CTA's item range.  Items are walked in order, so the position (split, group, layer, request)
// advances by counting, and everything that depends on the request alone (its batch metadata, tile counts) is computed
// when the request changes: per item there is no load from global memory.  A role thread that stalls at every item
// boundary stalls the pipeline behind it.
struct Walk {
    const TcParams &p;
    int w, w1, split, l, G, b, chunk;
    int64_t key;
    UnitInfo req;  // metadata of request `req.b` (-1: none read yet); l and G are not kept here
    int k_tiles, tps, n_chunks;
    Rows R;

    __device__ Walk(const TcParams &tp, int w0, int end) : p(tp), w(w0), w1(end), chunk(0) {
        const int units = p.mv.L * p.mv.G;
        split = w0 % p.splits;
        key = w0 / p.splits;
        const int unit = (int)(key % units);
        b = (int)(key / units);
        l = unit / p.mv.G;
        G = unit % p.mv.G;
        req.b = -1;
    }
    __device__ void next_unit() {  // past the splits of this unit that the CTA holds
        w += p.splits - split;
        chunk = 0;
        split = 0;
        ++key;
        if (++G == p.mv.G) {
            G = 0;
            if (++l == p.mv.L) {
                l = 0;
                ++b;
            }
        }
    }
    // `empties`: also stop (with R.rows = 0) at units of requests without prompt rows.
    __device__ bool next(Stop &s, bool empties, bool report) {
        for (; w < w1; next_unit()) {
            if (req.b != b) {
                req = unit_info(p.mv, p.bv, 0, b);
                k_tiles = n_key_tiles(req);
                tps = (k_tiles + p.splits - 1) / p.splits;  // key tiles per split
                n_chunks = max(1, (padded_rows(req.n_q, p.mv.hpg) + kMaxRows - 1) / kMaxRows);
                R = make_rows(req.n_q, p.mv.hpg, 0);
                if (!req.ok && report) atomicOr(p.status, FINCH_DEV_BAD_BATCH);
            }
            s.n_splits = min(p.splits - split, w1 - w);
            s.t0 = split * tps;
            s.t1 = min(k_tiles, s.t0 + s.n_splits * tps);
            if (!req.ok || s.t0 >= s.t1 || (req.n_q == 0 && !empties)) continue;
            s.u = req;
            s.u.l = l;
            s.u.G = G;
            s.R = n_chunks == 1 ? R : make_rows(req.n_q, p.mv.hpg, chunk);
            s.split = split;
            s.chunk = chunk;
            s.key = key;
            s.q_key = key * n_chunks + chunk + ((int64_t)b << 48);
            if (++chunk == n_chunks) next_unit();
            return true;
        }
        return false;
    }
};

// MASK: the batch gives every query row a number of candidates it attends to (causal rows); both sweeps then mask
// the (row, key) pairs beyond it.  The unmasked instantiation contains none of that code.
template <int MODE, int D, bool MASK>
__global__ void __launch_bounds__(kTcThreads, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap q_big, const __grid_constant__ CUtensorMap q_small,
                const __grid_constant__ CUtensorMap cache_map, const __grid_constant__ CUtensorMap chunk_map, TcParams p) {
    extern __shared__ uint8_t smem_raw[];
    const Cta c = cta_layout(smem_raw, (D / 64) * kSlabBytes, p.q_tiles, p.rows_alloc, p.stages);
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp-uniform for the compiler
    const uint32_t tmem = cta_setup(c, kSoftmaxWarps);
    // Barriers and tensor memory are set up; what follows reads what earlier kernels of the stream wrote.  The
    // second sweep's loads and MMAs read only the step's inputs, which were complete before the first sweep began;
    // what its immediate predecessors produce (the merged row statistics) is read by the softmax warps alone, so
    // only they (and the writer of the scores) wait, and the tensor pipe already fills the accumulators while the
    // statistics are being merged.
    if (MODE == kLse || warp >= 3) {
        dependency_wait();
        // The second sweep does not let its successor in: the selection's CTAs would settle on the first SMs that are free, or
        // beside CTAs that still compute (a step of 16 requests of 4K-32K tokens 6385 us with, 6190 without; 2 requests of 47
        // candidates on 28 x 2 units 47.3 and 37.1).
        if (MODE == kLse) dependents_may_launch();
    }
    // this CTA's contiguous range of work items
    const int w0 = p.bounds ? p.bounds[blockIdx.x] : (int)((int64_t)blockIdx.x * p.n_items / gridDim.x);
    const int w1 = p.bounds ? p.bounds[blockIdx.x + 1] : (int)((int64_t)(blockIdx.x + 1) * p.n_items / gridDim.x);
    Walk walk(p, w0, w1);
    Stop s;
    bool ok = true;
    int64_t q_key = -1;
    TileRing ring{p.q_tiles};

    if (warp == 0) {
        if (lane == 0) {
            prefetch_tensormap(&q_big);
            prefetch_tensormap(&q_small);
            prefetch_tensormap(&cache_map);
            prefetch_tensormap(&chunk_map);
        }
        __syncwarp();
        Producer<D, true, MODE == kLse> role{c, &q_big, &q_small, &cache_map, &chunk_map, mv.hpg, bv.total_q};
        while (ok && walk.next(s, false, lane == 0)) {
            ok = role.segment(s.u, s.R, s.t0, s.t1, q_key != s.q_key ? ring.take(s.R.n_qt) : -1);
            q_key = s.q_key;
        }
        role.drain();
    } else if (warp == 1) {
        Issuer<D> role(c, tmem);
        int base = 0;
        bool more = walk.next(s, false, false);
        while (ok && more) {
            const Rows R = s.R;
            const int t0 = s.t0, t1 = s.t1;
            const int64_t key = s.q_key;
            more = walk.next(s, false, false);
            const bool reload = q_key != key, release = more && s.q_key != key;
            q_key = key;
            if (reload) base = ring.take(R.n_qt);
            ok = MODE == kLse ? role.lse_segment(R, t0, t1, base, reload, release)
                              : role.colsum_segment(R, t0, t1, base, reload, release);
        }
    } else if (warp == 2) {
        PadCleaner<D> role{c};
        while (ok && walk.next(s, false, false)) {
            if (q_key == s.q_key) continue;
            q_key = s.q_key;
            const int base = ring.take(s.R.n_qt);
            if (pads_hold_rows(s.u, s.R, bv.total_q)) ok = role.clear(s.R, base);
        }
    } else if (warp == 3) {
        if (MODE == kColsum) {
            SumWriter role{c, lane};
            const int64_t cand = (int64_t)bv.total_cache + bv.total_chunk;
            while (ok && walk.next(s, true, false)) {
                float *out = p.unit_scores + ((int64_t)s.u.l * mv.G + s.u.G) * cand + s.u.cache0 + s.u.chunk0;
                if (s.u.n_q == 0)
                    role.zeros(s.u, s.t0, s.t1, out);
                else
                    ok = role.segment(s.u, s.R, s.t0, s.t1, out, s.chunk > 0);
            }
        }
    } else if (warp >= kCtlWarps) {
        Softmax<MASK> role(c, tmem, mv.scale * kLog2e);
        int epoch = 0;
        while (ok && walk.next(s, false, false)) {
            const UnitInfo &u = s.u;
            const Rows &R = s.R;
            if (MODE == kLse) {
                uint32_t live = 0;  // bit qb: this thread's row of query tile qb is a prompt row
                int lim[kQTiles];   // masked variant: candidates that row attends to
#pragma unroll
                for (int qb = 0; qb < kQTiles; ++qb) {
                    lim[qb] = 0;
                    const int row = role.row_of(R, qb);
                    if (qb < R.n_qt && row_live(R, row)) {
                        live |= 1u << qb;
                        if (MASK) lim[qb] = max(0, min(u.N, bv.row_limit[u.q0 + (R.r0 + row) % R.rp]));
                    }
                }
                typename Softmax<MASK>::RowStats st;
                if (!(ok = role.lse_segment(u, R, s.t0, s.t1, live, lim, st))) break;
                // the stop's statistics stand at its first split, nothing at the others
                float2 *parts = p.partial + (s.key * p.splits + s.split) * kGroups * p.slots + R.r0;
                role.store_stats(R, st, live, parts, p.slots, false);
                for (int i = 1; i < s.n_splits; ++i) role.store_stats(R, st, live, parts + (int64_t)i * kGroups * p.slots, p.slots, true);
            } else {
                // The merged statistics of the resident rows are staged once per CTA, every softmax warp its share, into
                // one of two buffers; a warp that has passed the barrier of epoch e has seen all warps finish epoch
                // e - 1, so the buffer of epoch e + 1 (= that of e - 1) is free by then.
                if (q_key != s.q_key) {
                    q_key = s.q_key;
                    float2 *stats = c.stats + (epoch & 1) * p.rows_alloc;
                    int *limits = c.limits + (epoch & 1) * p.rows_alloc;
                    int2 *bounds = c.bounds + (epoch & 1) * (p.rows_alloc / 16);
                    for (int r = threadIdx.x - kCtlWarps * 32; r < R.n_qt * kRows; r += kSoftmaxWarps * 32) {
                        float2 out = make_float2(0.f, 0.f);
                        int limit = 0;
                        if (row_live(R, r)) {
                            const int h = (R.r0 + r) / R.rp, pr = R.r0 + r - h * R.rp;
                            out = p.merged[((int64_t)u.l * mv.Hq + u.G * mv.hpg + h) * bv.total_q + u.q0 + pr];
                            if (MASK) limit = max(0, min(u.N, bv.row_limit[u.q0 + pr]));
                        }
                        stage_row(stats, r, out);
                        if (MASK) {
                            limits[r] = limit;
                            // the least and the most of every 16 rows; a row that weighs nothing does not count
                            int lo = row_live(R, r) ? limit : INT_MAX, hi = limit;
#pragma unroll
                            for (int d = 1; d < 16; d <<= 1) {
                                lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
                                hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
                            }
                            if (r % 16 == 0) bounds[r / 16] = make_int2(lo, hi);
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&c.stats_ready[0]);
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&c.stats_ready[0], epoch & 1, c.abort_flag)))) break;
                    ++epoch;
                }
                ok = role.colsum_segment(u, R, s.t0, s.t1, c.stats + ((epoch - 1) & 1) * p.rows_alloc,
                                         c.limits + ((epoch - 1) & 1) * p.rows_alloc,
                                         c.bounds + ((epoch - 1) & 1) * (p.rows_alloc / 16));
            }
        }
    }
    cta_teardown(c, tmem, p.status);
}

// With several requests in the batch the items differ in size (accumulators = key tiles x query tiles of their
// request), so equal item counts per CTA would leave the grid waiting for the CTAs that drew the long prompts and
// large caches.  This one-block kernel sums the work per request (items are ordered request-major, and all items
// of a request cost about the same), then gives every CTA of the persistent grid a contiguous item range of about
// equal work: bounds[i] = the item at which the running work passes i / n_ctas of the total.
__global__ void __launch_bounds__(1024)
plan_items_kernel(TcParams p, int *bounds, int n_ctas) {
    __shared__ unsigned long long warp_sum[32];
    __shared__ unsigned long long carry_s;
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    dependency_wait();
    dependents_may_launch();
    const unsigned long long ipr = (unsigned long long)mv.L * mv.G * p.splits;  // items per request
    if (tid == 0) {
        carry_s = 0;
        p.work_prefix[0] = 0;
    }
    __syncthreads();
    for (int base = 0; base < bv.batch; base += 1024) {
        const int b = base + tid;
        unsigned long long cost = 0;
        if (b < bv.batch) {
            const UnitInfo u = unit_info(mv, bv, 0, b);
            if (u.ok && u.n_q > 0 && u.N > 0) {
                // accumulators of one split; an accumulator of few rows costs about half of a full one, a key tile
                // with a single accumulator is bound by its load, and an item (a query load) costs about two more
                const int rows = padded_rows(u.n_q, mv.hpg), rest = rows % kRows;
                const int quarters = rows / kRows * 4 + (rest == 0 ? 0 : (rest <= 64 ? 2 : 4));
                cost = ipr * (unsigned long long)((n_key_tiles(u) + p.splits - 1) / p.splits * max(quarters, 5) + 8);
            }
        }
        unsigned long long incl = cost;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long up = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += up;
        }
        if (lane == 31) warp_sum[wid] = incl;
        __syncthreads();
        unsigned long long before = carry_s;
        for (int w = 0; w < wid; ++w) before += warp_sum[w];
        if (b < bv.batch) p.work_prefix[b + 1] = before + incl;
        __syncthreads();
        if (tid == 1023) carry_s = before + incl;
        __syncthreads();
    }
    const unsigned long long total = carry_s;
    for (int i = tid; i <= n_ctas; i += 1024) {
        int item;
        if (i == 0) {
            item = 0;
        } else if (i == n_ctas || total == 0) {
            item = p.n_items;
        } else {
            const unsigned long long target = total / n_ctas * i + total % n_ctas * i / n_ctas;
            int lo = 0, hi = bv.batch - 1;  // the last request whose prefix is <= target
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (p.work_prefix[mid] <= target) lo = mid; else hi = mid - 1;
            }
            const unsigned long long span = p.work_prefix[lo + 1] - p.work_prefix[lo];
            const unsigned long long into = span ? (target - p.work_prefix[lo]) * ipr / span : 0;
            item = (int)((unsigned long long)lo * ipr + (into < ipr ? into : ipr));
        }
        bounds[i] = item;
    }
}

// Merge the partial statistics of every prompt row -- per key split, softmax group and copy of the row -- in a fixed order
// into the pair the column pass uses: weights are exp2(s2 - R) * w with R = M + floor(log2 Z) and
// w = 2^floor(log2 Z) / Z in (1/2, 1], so the exponent never exceeds a few units whatever reference the parts were
// summed against.
__global__ void __launch_bounds__(128)
merge_stats_kernel(TcParams p) {
    const ModelView &mv = p.mv;
    const BatchView &bv = p.bv;
    dependents_may_launch();  // before the wait: the second sweep's CTAs may take over SMs as the first sweep's retire
    dependency_wait();
    const int h = blockIdx.y % mv.Hq, l = blockIdx.y / mv.Hq;
    const UnitInfo u = unit_info(mv, bv, l * mv.G + h / mv.hpg, blockIdx.z);
    if (!u.ok || u.n_q == 0 || u.N == 0) return;
    const int pr = blockIdx.x * 128 + threadIdx.x;
    if (pr >= u.n_q) return;
    const int rp = (u.n_q + kRowPad - 1) / kRowPad * kRowPad, r = (h % mv.hpg) * rp + pr;
    const Rows R = make_rows(u.n_q, mv.hpg, r / kMaxRows);
    const int qb = r % kMaxRows / kRows;
    const int k_tiles = n_key_tiles(u);
    const int tps = (k_tiles + p.splits - 1) / p.splits;
    const int64_t row = ((int64_t)l * mv.Hq + h) * bv.total_q + u.q0 + pr;
    const int64_t key = (int64_t)blockIdx.z * mv.L * mv.G + l * mv.G + h / mv.hpg;
    const float2 *src = p.partial + key * p.splits * kGroups * p.slots + r;
    const Parts parts(R, qb);
    const int n = parts.count((k_tiles + tps - 1) / tps);  // splits that hold key tiles
    float M = -INFINITY, Z = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 8) {  // eight loads in flight, folded in order
        float2 part[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) part[i] = i0 + i < n ? src[parts.at(i0 + i, p.slots)] : make_float2(0.f, 0.f);
        merge_parts(part, M, Z);
    }
    if (bv.self_lse) merge_self_term(bv.self_lse[row], M, Z);  // the keys the row attends to besides the candidates
    float2 out = merged_pair(M, Z);
    if (bv.row_limit && bv.row_norm)  // per-row normalisation: times the fraction of the candidates the row sees
        out.y *= (float)max(0, min(u.N, bv.row_limit[u.q0 + pr])) / (float)u.N;
    p.merged[row] = out;
    if (p.row_lse) p.row_lse[row] = merged_lse(M, Z);
}

// ------------------------------------------------------------------------------------------------ host side

// Key splits per unit, at least one key tile each and at most kScoreMaxSplits: the smallest count whose grid fills whole
// waves of SMs best, every item (unit, request, split) costing the same.  Several requests' items differ, and CTAs take
// ranges of about equal work: where there are enough of them eight items to a CTA are fine enough (9 requests of 16 units:
// 144 items on 148 SMs left the grid waiting for the longest prompts, 0.144 ms against 0.120); few units would only load
// their queries on more CTAs (2 requests of 16 units: 46 us with 4 splits, 66 with 8).
int choose_splits(int units, int batch, int key_tiles, int sm_count) {
    const int most = min(kScoreMaxSplits, key_tiles);
    if (batch > 1 && 2 * units * batch >= sm_count) {
        units *= batch;
        // where every SM has a unit already, a split of fewer than three key tiles is mostly its queries and its statistics (23
        // requests of 98 candidates on 4 x 8 units: 48 us with a split to each of two tiles, 44 with none)
        const int worth = units >= sm_count ? max(1, key_tiles / 3) : key_tiles;
        return max(1, min(min(most, worth), (8 * sm_count + units - 1) / units));
    }
    units *= batch;
    int best = 1;
    double best_eff = 0.0;
    for (int s = 1; s <= most; ++s) {
        const double waves = (double)units * s / sm_count;
        const double eff = waves / (double)((long long)waves + (waves > (long long)waves ? 1 : 0));
        if (eff > best_eff * 1.05) {
            best_eff = eff;
            best = s;
        }
    }
    return best;
}

template <int D, bool MASK>
cudaError_t launch_d(const Ctx &ctx, const CUtensorMap &qb, const CUtensorMap &qs, const CUtensorMap &cm, const CUtensorMap &hm,
                     TcParams p, float *scores, cudaStream_t stream) {
    constexpr int kTileBytes = (D / 64) * kSlabBytes;
    const ModelView &mv = p.mv;  // the scoring view
    const BatchView &bv = p.bv;
    p.rows_alloc = min(kMaxRows, p.slots);
    p.q_tiles = min(kQTiles, p.rows_alloc / kRows + 1);  // the next item's queries arrive while this one's are in use
    if (p.rows_alloc / kRows == 2) p.q_tiles = kQTiles;
    p.stages = kMaxStages;
    while (p.stages > 2 && cta_smem(kTileBytes, p.q_tiles, p.rows_alloc, p.stages, MASK) > kSmemLimit) --p.stages;
    const int smem = cta_smem(kTileBytes, p.q_tiles, p.rows_alloc, p.stages, MASK);
    cudaError_t e = cudaSuccess;
    const int bit = kSmemTc + (D == 128) * 2 + MASK;
    if (!ctx.smem_ready(bit)) {
        e = cudaFuncSetAttribute(score_tc_kernel<kLse, D, MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(score_tc_kernel<kColsum, D, MASK>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
        if (e != cudaSuccess) return e;
        ctx.smem_set(bit);
    }
    p.n_items = p.splits * mv.L * mv.G * bv.batch;
    const int sms = ctx.sm_count > 0 ? ctx.sm_count : 148;
    dim3 grid(p.n_items < sms ? p.n_items : sms);  // persistent: one CTA per SM walks a contiguous range of items
    if (bv.batch > 1 && (int)grid.x < kPlanBoundsInts) {  // requests of different sizes: ranges of equal work
        int *bounds = (int *)(p.work_prefix + bv.batch + 1);
        e = launch_chained(plan_items_kernel, dim3(1), dim3(1024), 0, stream, p, bounds, (int)grid.x);
        if (e != cudaSuccess) return e;
        p.bounds = bounds;
        ctx.launches += 1;
    }
    e = launch_chained(score_tc_kernel<kLse, D, MASK>, grid, dim3(kTcThreads), smem, stream, qb, qs, cm, hm, p);
    if (e != cudaSuccess) return e;
    dim3 mgrid((bv.max_q + 127) / 128, mv.L * mv.Hq, bv.batch);
    e = launch_chained(merge_stats_kernel, mgrid, dim3(128), 0, stream, p);
    if (e != cudaSuccess) return e;
    e = launch_chained(score_tc_kernel<kColsum, D, MASK>, grid, dim3(kTcThreads), smem, stream, qb, qs, cm, hm, p);
    ctx.launches += 3;
    if (e != cudaSuccess || ctx.model.G == mv.G) return e;
    return launch_sum_heads(ctx, mv, bv, p.unit_scores, scores, ctx.model.G, ctx.model.kvpg, stream);
}

int slots_of(const ModelView &mv, const BatchView &bv) {  // padded query rows of the longest unit, whole tiles
    return (padded_rows(bv.max_q, mv.g) + kRows - 1) / kRows * kRows;
}

// Scratch (float2 entries) besides the partial row statistics: item plan, merged rows, per-KV-head scores.
size_t scratch_rest(const ModelView &mv, const BatchView &bv) {
    const size_t rows = (size_t)mv.L * mv.Hq * (size_t)bv.total_q;
    const size_t cand = (size_t)mv.L * mv.Hkv * ((size_t)bv.total_cache + bv.total_chunk);
    return rows + (cand + 1) / 2 + (size_t)bv.batch + 1 + kPlanBoundsInts / 2;
}

}  // namespace

bool score_tc_supported(const Ctx &ctx) {
    return ctx.cfg.dtype == FINCH_BF16 && (ctx.model.d == 64 || ctx.model.d == 128);
}

// Scratch (float2 entries) of the two-launch tensor-core path: the least, with one key split, and what it would like.
size_t score_tc_scratch_min(const Ctx &ctx, const BatchView &bv) {
    const ModelView &mv = ctx.model;
    return (size_t)bv.batch * mv.L * mv.Hkv * kGroups * slots_of(mv, bv) + scratch_rest(mv, bv);
}
size_t score_tc_scratch(const Ctx &ctx, const BatchView &bv) {
    const ModelView &mv = ctx.model;
    const int key_tiles = (bv.max_cache + kRows - 1) / kRows + (bv.max_chunk + kRows - 1) / kRows;
    if (bv.batch == 0 || key_tiles == 0) return 0;
    const size_t splits = choose_splits(mv.L * mv.Hkv, bv.batch, key_tiles, ctx.sm_count > 0 ? ctx.sm_count : 148);
    return splits * bv.batch * mv.L * mv.Hkv * kGroups * slots_of(mv, bv) + scratch_rest(mv, bv);
}

// What it would like for no batch within these bounds to want more: key splits times requests grow as bounds shrink.
size_t score_tc_scratch_bound(const Ctx &ctx, const BatchView &bv) {
    const ModelView &mv = ctx.model;
    const int key_tiles = (bv.max_cache + kRows - 1) / kRows + (bv.max_chunk + kRows - 1) / kRows;
    if (bv.batch == 0 || key_tiles == 0) return 0;
    const size_t sms = ctx.sm_count > 0 ? ctx.sm_count : 148, units = (size_t)mv.L * mv.Hkv, items = units * bv.batch;
    const size_t most = min(kScoreMaxSplits, key_tiles);
    size_t one = 1;  // splits of a single request
    for (size_t t = 1; t <= most; ++t) one = max(one, (size_t)choose_splits((int)units, 1, (int)t, (int)sms));
    // of several: choose_splits, with 8 x SMs rounded up to whole splits, or up to half the SMs' items with any number of splits
    size_t n = units * one;
    if (bv.batch > 1) n = max(n, min(most * items, max(8 * sms + items, most * (sms / 2 + 1))));
    return n * kGroups * slots_of(mv, bv) + scratch_rest(mv, bv);
}

// `scratch` holds `capacity` float2 entries; the key-split count is limited so that everything fits.  Returns
// cudaErrorNotSupported (and launches nothing) when it does not, or when the tensors cannot be described to the TMA
// unit; the caller then uses the warp-level path for every request.
cudaError_t launch_score_tc(const Ctx &ctx, const TensorView &q, const TensorView &cache_k, const TensorView &chunk_k,
                            const BatchView &bv, float *scores, float2 *scratch, size_t capacity, float *row_lse,
                            cudaStream_t stream) {
    // Scoring works per KV head whatever the selection groups are: a query head only ever meets its own KV head's
    // keys.  With one selection group per layer the heads' column sums are added afterwards.
    ModelView mv = ctx.model;
    mv.G = mv.Hkv;
    mv.hpg = mv.g;
    mv.kvpg = 1;
    if (mv.L * mv.G == 0 || bv.batch == 0 || bv.max_q == 0 || bv.max_cache + bv.max_chunk == 0) return cudaSuccess;
    // scratch layout (float2 units): item plan | merged row statistics | per-KV-head scores | partial row statistics
    const size_t rows = (size_t)mv.L * mv.Hq * (size_t)bv.total_q;
    const size_t plan = (size_t)bv.batch + 1 + kPlanBoundsInts / 2;  // 64-bit work prefix, then the CTA bounds
    const size_t cand = (size_t)mv.L * mv.Hkv * ((size_t)bv.total_cache + bv.total_chunk);
    const size_t rest = scratch_rest(mv, bv);
    const int slots = slots_of(mv, bv);
    const size_t per_split = (size_t)bv.batch * mv.L * mv.Hkv * kGroups * slots;
    if (rows == 0 || capacity < rest + per_split) return cudaErrorNotSupported;
    CUtensorMap qb, qs, cm, hm;
    if (!make_map(&qb, q, mv.d, bv.total_q, mv.Hq, mv.L, kBigBox)) return cudaErrorNotSupported;
    if (!make_map(&qs, q, mv.d, bv.total_q, mv.Hq, mv.L, kRowPad)) return cudaErrorNotSupported;
    const bool have_cache = bv.max_cache > 0, have_chunk = bv.max_chunk > 0;
    if (have_cache && !make_map(&cm, cache_k, mv.d, bv.total_cache, mv.Hkv, mv.L, kRows)) return cudaErrorNotSupported;
    if (have_chunk && !make_map(&hm, chunk_k, mv.d, bv.total_chunk, mv.Hkv, mv.L, kRows)) return cudaErrorNotSupported;
    if (!have_cache) cm = hm;  // never dereferenced: no request has cache tiles
    if (!have_chunk) hm = cm;
    const int key_tiles = (bv.max_cache + kRows - 1) / kRows + (bv.max_chunk + kRows - 1) / kRows;
    const int most = (int)min((size_t)kScoreMaxSplits, (capacity - rest) / per_split);  // splits the scratch has room for
    TcParams p{};
    p.mv = mv;
    p.bv = bv;
    p.row_lse = row_lse;
    p.status = ctx.d_status;
    p.slots = slots;
    p.splits = min(most, choose_splits(mv.L * mv.G, bv.batch, key_tiles, ctx.sm_count > 0 ? ctx.sm_count : 148));
    p.work_prefix = (unsigned long long *)scratch;
    p.merged = scratch + plan;
    p.unit_scores = ctx.model.G == mv.G ? scores : (float *)(p.merged + rows);
    p.partial = p.merged + rows + (cand + 1) / 2;
    if (bv.row_limit)  // causal query rows: the masked instantiation
        return mv.d == 64 ? launch_d<64, true>(ctx, qb, qs, cm, hm, p, scores, stream)
                          : launch_d<128, true>(ctx, qb, qs, cm, hm, p, scores, stream);
    return mv.d == 64 ? launch_d<64, false>(ctx, qb, qs, cm, hm, p, scores, stream)
                      : launch_d<128, false>(ctx, qb, qs, cm, hm, p, scores, stream);
}

}  // namespace finch
