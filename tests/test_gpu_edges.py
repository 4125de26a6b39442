"""GPU parity at the sizes where the kernels' tilings and dispatch rules change: row padding, copies of a short query tile,
query chunks, ranges of one unit exchanged through a cluster or through global memory, candidates per selection kernel,
row blocks of the compaction, key splits of the warp-level scoring.  Against the fp64 oracle, with the harness's tolerance
(max(1e-3 relative, 1e-5 absolute) per score, everything else exact)."""
import numpy as np
import pytest

import oracle
from paper_2408_00167_b200 import binding as fb
from paper_2408_00167_b200 import build as fbuild
from paper_2408_00167_b200 import workloads as wl
from parity_harness import GpuStep, check_parity, oracle_scores, to_device, to_host
from test_gpu_configs import _select_only

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()
    fb.load()


def _check(layers, Hq, Hkv, d, reqs, dtype="bf16", group_mode=0):
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=layers, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, dtype=dtype,
                    group_mode=group_mode, planted_frac=0.02, requests=tuple(wl.Request(*r) for r in reqs))
    st = wl.steady_state(cfg, list(range(layers)), step=1)
    g = GpuStep(cfg, st, layers)
    try:
        plan = fb.finch_score_plan(g.ctx, g.batch)
        g.run_parts()
        assert g.status() == 0
        res = g.results()
        for b in range(cfg.batch):      # every candidate has a number
            lo = int(st["cache_off"][b] + st["chunk_off"][b])
            hi = lo + int(st["cache_len"][b] + st["chunk_off"][b + 1] - st["chunk_off"][b])
            assert np.isfinite(res["scores"][:, :, lo:hi]).all()
        ref, ref_lse = oracle_scores(cfg, st, threads=oracle.max_threads(), want_lse=True)
        check_parity(cfg, st, res, ref)
        # the log of a sum of exponentials of fp32 logits: a few 2^-24 of the largest logit (below 2^6 here)
        np.testing.assert_allclose(res["row_lse"], ref_lse, rtol=1e-5, atol=2e-5)
    finally:
        g.close()
    return plan


@pytest.mark.parametrize("heads,n_q", [(1, 1), (1, 32), (1, 33), (1, 65), (1, 128), (2, 65), (4, 37), (4, 96), (4, 128)])
def test_query_rows_around_the_tile_sizes(heads, n_q):
    """Padded rows per KV head from 8 to 512: one to four query tiles, a last one of 32, 64 and 128 rows."""
    path, _ = _check(1, 2 * heads, 2, 128, [(n_q, 9999, 300, 200)])
    assert path == fb.FINCH_SCORE_ONE_KERNEL


@pytest.mark.parametrize("layers,Hkv,cache,chunk,window", [
    (1, 2, 1, 127, 1),        # two tiles, one candidate in the first
    (1, 8, 512, 512, 2),      # four ranges of two tiles: a cluster
    (1, 8, 2048, 2048, 4),    # eight ranges
    (5, 8, 2030, 2032, None),  # three ranges a unit, the last one shorter
    (20, 8, 640, 256, 7),     # whole units in two windows, the second one half empty
    (19, 16, 1024, 1024, None),   # several windows whose ranges meet across CTAs
])
def test_ranges_of_a_unit(layers, Hkv, cache, chunk, window):
    path, w = _check(layers, Hkv, Hkv, 64, [(24, 99999, chunk, cache)])
    assert path == fb.FINCH_SCORE_ONE_KERNEL and (window is None or w == window)


@pytest.mark.parametrize("n_q,heads", [(129, 4), (145, 4), (513, 1)])
def test_query_chunks_and_pad_rows_of_neighbouring_requests(n_q, heads):
    """More than 512 padded rows in chunks; requests whose pad rows are the next request's rows."""
    path, _ = _check(2, 2 * heads, 2, 128, [(n_q, 9999, 200, 150), (7, 9999, 140, 260), (n_q - 3, 9999, 100, 129)])
    assert path == fb.FINCH_SCORE_TWO_LAUNCH


@pytest.mark.parametrize("n", [63, 64, 65, 2047, 2048, 2049, 4095, 8191, 8192, 8193])
@pytest.mark.parametrize("kind", ["spread", "one_value", "two_values", "outlier"])
def test_select_at_the_limits_of_its_kernels(n, kind):
    rng = np.random.default_rng(n)
    L, G = 2, 2
    s = rng.random((L, G, n), dtype=np.float32)
    if kind == "one_value":
        s[:] = 0.25                                   # a single key: the first round's bin holds everything
    elif kind == "two_values":
        s = np.where(s < 0.5, np.float32(0.5), np.nextafter(np.float32(0.5), np.float32(1))).astype(np.float32)
    elif kind == "outlier":
        s = (1 + s * 1e-4).astype(np.float32)         # all but one key in one bin of the first round
        s[:, :, n // 3] = 1e30
    for r in (1, n // 2, n - 1):
        kept, out_len = _select_only(s, [n], [n], [0], [r], L, G)
        assert out_len.tolist() == [r]
        for l in range(L):
            for g in range(G):
                np.testing.assert_array_equal(kept[l, g, :r], oracle.select_unit(s[l, g].astype(np.float64), r))


@pytest.mark.parametrize("Hq,Hkv,n_q,cache,chunk,d", [(8, 8, 16, 256, 256, 64), (8, 2, 17, 64, 1, 96), (8, 2, 32, 130, 65, 32),
                                                     (8, 2, 33, 63, 64, 128), (4, 4, 65, 700, 1400, 64)])
def test_warp_level_scoring_tiles_and_splits(Hq, Hkv, n_q, cache, chunk, d):
    _check(1, Hq, Hkv, d, [(n_q, 9999, chunk, cache)], dtype="f32")


def test_causal_blocks_that_see_all_none_or_part_of_their_keys():
    """Query rows in blocks with one limit each: nothing, one key, the tile edges and their neighbours, everything."""
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=2, n_q_heads=2, n_kv_heads=1, head_dim=128, dtype="bf16", planted_frac=0.03,
                    requests=(wl.Request(280, 9999, 300, 212),))
    st = wl.steady_state(cfg, [0, 1], step=2)
    N = 512
    limit = np.repeat(np.array([0, 1, 31, 32, 33, 127, 128, 129, 211, 212, 213, 383, 384, N, N + 9], np.int32), 19)[:280]
    limit[-40:] = np.arange(N - 40, N)                      # a ragged staircase at the end
    g = GpuStep(cfg, st, 2, row_limit=limit)
    try:
        g.run_parts()
        assert g.status() == 0
        res = g.results()
        ref, ref_lse = oracle_scores(cfg, st, want_lse=True, row_limit=limit)
        check_parity(cfg, st, res, ref)
        finite = np.isfinite(ref_lse)
        np.testing.assert_allclose(res["row_lse"][finite], ref_lse[finite], rtol=1e-5, atol=2e-5)
        assert np.all(np.isneginf(res["row_lse"][~finite]))
    finally:
        g.close()


@pytest.mark.parametrize("rope_theta", [0.0, 10000.0])
@pytest.mark.parametrize("L,Hkv,budget", [(1, 1, 1), (1, 2, 17), (1, 4, 255), (8, 8, 257), (32, 32, 600)])
def test_compact_row_blocks(L, Hkv, budget, rope_theta):
    """Budgets around the row blocks of one CTA (16 to 256 rows, by how many KV heads share the chip)."""
    import torch
    rng = np.random.default_rng(budget)
    d, c, m = 64, 400, 300
    mk = lambda n: wl.to_storage(rng.standard_normal((L, Hkv, n, d)).astype(np.float32), "bf16")
    ck, cv, hk, hv = mk(budget + c), mk(budget + c), mk(m), mk(m)
    cache_off, chunk_off = wl.offsets([budget + c]), wl.offsets([m])
    cpos = rng.integers(0, 1000, size=(L, Hkv, budget + c)).astype(np.int32)
    hpos = rng.integers(1000, 2000, size=m).astype(np.int32)
    scores = rng.random((L, Hkv, budget + c + m))
    kept, out_len = oracle.select(scores, chunk_off=chunk_off, cache_off=cache_off, cache_len=[c], budget=[budget])
    kw = dict(n_kv_heads=Hkv, head_dim=d, group_mode=0, chunk_off=chunk_off, cache_off=cache_off, cache_len=[c])
    if rope_theta:
        kw.update(rope_theta=rope_theta, rope_pairing=0)
    want_k, want_v, want_p = oracle.compact("bf16", kept, out_len, ck, cv, cpos, hk, hv, hpos, **kw)
    batch = fb.make_batch(wl.offsets([1]), chunk_off, cache_off, [c], [budget])
    ctx = fb.finch_ctx_create(L, Hkv, Hkv, d, fb.FINCH_BF16, 0, max_batch=1, max_prompt=1, max_candidates=2048,
                              rope_theta=rope_theta)
    try:
        dev = lambda a: to_device(a, "bf16")
        out_k, out_v = dev(np.zeros_like(ck)), dev(np.zeros_like(cv))
        out_pos = torch.full((L, Hkv, budget + c), -1, dtype=torch.int32, device="cuda")
        fb.finch_compact(ctx, torch.from_numpy(kept).cuda(), torch.from_numpy(out_len).cuda(), dev(ck), dev(cv),
                         torch.from_numpy(cpos).cuda(), dev(hk), dev(hv), torch.from_numpy(hpos).cuda(), batch,
                         out_k, out_v, out_pos)
        assert fb.finch_device_status(ctx) == 0
        np.testing.assert_array_equal(to_host(out_v, "bf16"), want_v)
        np.testing.assert_array_equal(out_pos.cpu().numpy(), want_p)
        if not rope_theta:
            np.testing.assert_array_equal(to_host(out_k, "bf16"), want_k)
        else:       # fp32 rotation: one unit in the last place of a bfloat16 (2^-8 relative to its binade's top) on near-ties
            got = wl.from_storage(to_host(out_k, "bf16"), "bf16").astype(np.float64)
            want = wl.from_storage(want_k, "bf16").astype(np.float64)
            row = np.sqrt((want ** 2).sum(axis=-1, keepdims=True))
            assert np.all(np.abs(got - want) <= np.abs(want) * 2.0 ** -7 + 2e-6 * row)
    finally:
        fb.finch_ctx_destroy(ctx)


@pytest.mark.parametrize("rope_theta", [0.0, 10000.0])
@pytest.mark.parametrize("layers,Hkv,reqs,dtype,group_mode,keep_all,d,one_launch", [
    (1, 8, [(16, 9999, 256, 256)], "f32", 0, False, 64, True),       # blocks of 16 rows
    (1, 8, [(20, 9999, 2048, 2048)], "bf16", 0, False, 64, True),    # the longest unit that is selected beside its copies
    (1, 8, [(20, 9999, 2049, 2048)], "bf16", 0, False, 64, False),   # one candidate more: two launches
    (12, 37, [(8, 9999, 70, 512)], "bf16", 0, False, 64, None),      # 444 blocks of 512 rows
    (12, 37, [(8, 9999, 70, 513)], "bf16", 0, False, 64, False),     # a row more: two launches
    (2, 4, [(9, 9999, 300, 77)], "bf16", 1, False, 64, True),        # one selection group per layer
    (1, 4, [(9, 9999, 33, 15), (5, 9999, 1, 90), (3, 9999, 64, 64)], "bf16", 0, False, 64, False),   # scored in two launches
    (1, 4, [(9, 9999, 33, 15), (5, 9999, 1, 90), (3, 9999, 64, 64)], "f32", 0, False, 64, True),     # several requests
    (2, 3, [(9, 9999, 70, 40), (5, 9999, 20, 0), (3, 9999, 600, 300)], "bf16", 0, False, 96, True),  # one with nothing to keep
    (2, 2, [(4, 9999, 200, 100), (7, 9999, 50, 33)], "f32", 1, False, 128, True),
    (2, 3, [(9, 9999, 90, 200)], "f32", 1, True, 64, True),          # a budget that keeps everything
])
def test_step_that_selects_and_copies_in_one_launch(layers, Hkv, reqs, dtype, group_mode, keep_all, d, one_launch, rope_theta):
    """finch_step against the oracle and, bit for bit, against the three calls it stands for; by the number of its kernels it is
    told whether the step took the one launch (None: that depends on how many of its CTAs an SM holds)."""
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=layers, n_q_heads=Hkv, n_kv_heads=Hkv, head_dim=d, dtype=dtype,
                    group_mode=group_mode, planted_frac=0.05, requests=tuple(wl.Request(*r) for r in reqs))
    st = wl.steady_state(cfg, list(range(layers)), step=1)
    if keep_all:
        st["cache_len"] = st["cache_len"] - np.diff(st["chunk_off"]).astype(st["cache_len"].dtype)
    runs, launches = [], []
    for parts in (False, True):
        g = GpuStep(cfg, st, layers)
        try:
            if rope_theta:
                c = g.batch.c
                fb.finch_ctx_destroy(g.ctx)
                g.ctx = fb.finch_ctx_create(layers, Hkv, Hkv, d, fb.FINCH_F32 if dtype == "f32" else fb.FINCH_BF16, group_mode,
                                            max_batch=len(reqs), max_prompt=c.max_q, max_candidates=c.max_cache + c.max_chunk,
                                            rope_theta=rope_theta)
            for _ in range(1 if parts else 2):
                before = fb.finch_launch_count(g.ctx)
                g.run_parts() if parts else g.run()
                count = fb.finch_launch_count(g.ctx) - before
            assert g.status() == 0
            runs.append(g.results())
            launches.append(count)
        finally:
            g.close()
    if one_launch is not None:
        assert launches[1] - launches[0] == int(one_launch)
    for name in ("kept_idx", "out_len", "out_pos", "out_k", "out_v"):
        np.testing.assert_array_equal(runs[0][name], runs[1][name], err_msg=name)
    if not rope_theta:
        check_parity(cfg, st, runs[0], oracle_scores(cfg, st, threads=oracle.max_threads()))


@pytest.mark.parametrize("layers,Hkv,n_q,cache,chunk", [(1, 2, 520, 100, 70), (3, 4, 513, 700, 129), (1, 1, 600, 2048, 2048)])
def test_single_request_scored_in_two_launches_selects_and_copies_in_one(layers, Hkv, n_q, cache, chunk):
    """More than 512 prompt rows per KV head: the step has one kernel less than its three calls, and their results."""
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=layers, n_q_heads=Hkv, n_kv_heads=Hkv, head_dim=64, planted_frac=0.05,
                    requests=(wl.Request(n_q, 9999, chunk, cache),))
    st = wl.steady_state(cfg, list(range(layers)), step=1)
    runs, launches = [], []
    for parts in (False, True):
        g = GpuStep(cfg, st, layers)
        try:
            assert fb.finch_score_plan(g.ctx, g.batch)[0] == fb.FINCH_SCORE_TWO_LAUNCH
            before = fb.finch_launch_count(g.ctx)
            g.run_parts() if parts else g.run()
            launches.append(fb.finch_launch_count(g.ctx) - before)
            assert g.status() == 0
            runs.append(g.results())
        finally:
            g.close()
    assert launches[1] - launches[0] == 1
    for name in ("kept_idx", "out_len", "out_pos", "out_k", "out_v"):
        np.testing.assert_array_equal(runs[0][name], runs[1][name], err_msg=name)


@pytest.mark.parametrize("layers,Hq,Hkv,n_q,cache,chunk,rope_theta", [
    (1, 2, 2, 40, 100, 40, 0.0),           # few rows
    (3, 8, 4, 300, 700, 129, 10000.0),     # 608 rows per KV head, kept keys rotated
    (2, 4, 1, 520, 300, 900, 0.0),         # five chunks of rows
])
def test_causal_request_selects_and_copies_in_one_launch(layers, Hq, Hkv, n_q, cache, chunk, rope_theta):
    """A single request with limits: finch_step has one kernel less than its three calls, their results, and the oracle's scores."""
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=layers, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=64, planted_frac=0.05,
                    requests=(wl.Request(n_q, 9999, chunk, cache),))
    st = wl.steady_state(cfg, list(range(layers)), step=1)
    limit = np.minimum(cache + 1 + np.arange(n_q), cache + chunk).astype(np.int32)
    runs, launches = [], []
    for parts in (False, True):
        g = GpuStep(cfg, st, layers, row_limit=limit)
        try:
            if rope_theta:
                fb.finch_ctx_destroy(g.ctx)
                g.ctx = fb.finch_ctx_create(layers, Hq, Hkv, 64, fb.FINCH_BF16, 0, max_batch=1, max_prompt=n_q,
                                            max_candidates=g.batch.c.max_cache + g.batch.c.max_chunk, rope_theta=rope_theta)
            assert fb.finch_score_plan(g.ctx, g.batch)[0] == fb.FINCH_SCORE_TWO_LAUNCH
            before = fb.finch_launch_count(g.ctx)
            g.run_parts() if parts else g.run()
            launches.append(fb.finch_launch_count(g.ctx) - before)
            assert g.status() == 0
            runs.append(g.results())
        finally:
            g.close()
    assert launches[1] - launches[0] == 1
    for name in ("kept_idx", "out_len", "out_pos", "out_k", "out_v"):
        np.testing.assert_array_equal(runs[0][name], runs[1][name], err_msg=name)
    if not rope_theta:
        check_parity(cfg, st, runs[0], oracle_scores(cfg, st, threads=oracle.max_threads(), row_limit=limit))


@pytest.mark.parametrize("fill", [float("nan"), 3e4])
@pytest.mark.parametrize("layers,n_q,extra,causal", [(1, 37, 3, False), (12, 9, 40, False), (1, 150, 1, False), (1, 257, 3, False),
                                                     (2, 37, 5, True)])
def test_rows_behind_the_requests_reach_no_score(layers, n_q, extra, causal, fill):
    """A query tensor with rows behind the last request's: they are no prompt rows, whatever they hold.  One kernel with one
    window and with several, halves of a KV head's queries, chunks of 512 rows in two launches (1056 padded rows), masked
    rows: bit for bit the scores of the tensor without them."""
    import torch
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=layers, n_q_heads=16, n_kv_heads=4, head_dim=64, planted_frac=0.02,
                    requests=(wl.Request(n_q, 9999, 300, 500),))
    st = wl.steady_state(cfg, list(range(layers)), step=1)
    limit = np.linspace(1, 800, n_q).astype(np.int32) if causal else None
    g = GpuStep(cfg, st, layers, row_limit=limit)
    try:
        g.run_parts()
        want, want_lse = g.scores.clone(), g.row_lse.clone()
        g.q = torch.cat([g.q, torch.full_like(g.q[:, :, :1], fill).expand(-1, -1, extra, -1)], dim=2)
        g.batch.c.total_q += extra
        if causal:
            g.batch.row_limit = torch.cat([g.batch.row_limit, torch.full_like(g.batch.row_limit[:1], 800).expand(extra)])
            g.batch.c.row_limit = g.batch.row_limit.data_ptr()
        g.row_lse = torch.zeros((layers, 16, n_q + extra), device="cuda")
        g.ws = torch.empty(fb.finch_workspace_bytes(g.ctx, g.batch), dtype=torch.uint8, device="cuda")
        g.run_parts()
        assert g.status() == 0 and g.guards_intact()
        np.testing.assert_array_equal(g.scores.cpu().numpy(), want.cpu().numpy())
        np.testing.assert_array_equal(g.row_lse[:, :, :n_q].cpu().numpy(), want_lse.cpu().numpy())
    finally:
        g.close()


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (96, "bf16")])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_key_that_is_no_number_voids_its_rows_whatever_the_key_split(d, dtype, bad):
    """Warp-level scoring: a row whose sum is NaN weighs nothing, also where the bad key lies in one of several key splits."""
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=1, n_q_heads=2, n_kv_heads=2, head_dim=d, dtype=dtype, planted_frac=0.02,
                    requests=(wl.Request(9, 9999, 200, 300),))
    st = wl.steady_state(cfg, [0], step=1)
    g = GpuStep(cfg, st, 1)
    try:
        g.run_parts()
        want, want_lse = g.scores.cpu().numpy().copy(), g.row_lse.cpu().numpy().copy()
        g.cache_k[0, 0, 100, 3] = bad
        g.run_parts()
        got, lse = g.scores.cpu().numpy(), g.row_lse.cpu().numpy()
        assert g.status() == 0
        np.testing.assert_array_equal(got[0, 1], want[0, 1])            # the other head
        np.testing.assert_array_equal(lse[0, 1], want_lse[0, 1])
        if np.isnan(bad):
            assert np.all(np.isneginf(lse[0, 0])) and np.isnan(got[0, 0, 100])
            assert np.all(np.delete(got[0, 0], 100) == 0)
        else:                                                            # a logit of -inf is a weight of 0, one of +inf voids the row
            up = st["q"][0, 0].reshape(9, d)[:, 3]
            up = wl.from_storage(up, dtype) > 0
            assert np.array_equal(np.isneginf(lse[0, 0]), up)
    finally:
        g.close()


@pytest.mark.parametrize("heads,rows", [(1, 23), (4, 9), (2, 70)])
def test_many_small_requests_do_not_see_their_neighbours(heads, rows):
    """Units of one or two query tiles and a few key tiles, many to a CTA; NaN in every third request's queries."""
    import torch
    rng = np.random.default_rng(rows)
    reqs = [wl.Request(int(rng.integers(1, rows + 1)), 9999, int(rng.integers(1, 140)), int(rng.integers(1, 140))) for _ in range(41)]
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=3, n_q_heads=4 * heads, n_kv_heads=4, head_dim=128, planted_frac=0.05,
                    requests=tuple(reqs))
    st = wl.steady_state(cfg, [0, 1, 2], step=1)
    g = GpuStep(cfg, st, 3)
    try:
        g.run_parts()
        assert g.status() == 0
        res = g.results()
        check_parity(cfg, st, res, oracle_scores(cfg, st, threads=oracle.max_threads()))
        for b in range(0, 41, 3):
            g.q[:, :, int(st["q_off"][b]):int(st["q_off"][b + 1])] = float("nan")
        g.run_parts()
        got = g.scores.cpu().numpy()
        for b in range(41):
            if b % 3:
                lo = int(st["cache_off"][b] + st["chunk_off"][b])
                hi = lo + int(st["cache_len"][b] + st["chunk_off"][b + 1] - st["chunk_off"][b])
                np.testing.assert_array_equal(got[:, :, lo:hi], res["scores"][:, :, lo:hi], err_msg=f"request {b}")
    finally:
        g.close()


@pytest.mark.parametrize("layers,Hkv,heads,d,n_q,cache,chunk", [
    (1, 2, 1, 128, 1, 1, 127),        # one window of one and of two key tiles: an issuer without a tile of its own
    (1, 2, 1, 64, 64, 300, 200),      # two key tiles to an accumulator, an odd number of tiles
    (1, 2, 1, 64, 65, 300, 200),      # the same with one
    (20, 8, 1, 128, 128, 640, 256),   # several windows of an odd number of tiles: the issuers swap tiles from window to window
    (20, 8, 4, 64, 16, 1000, 129),    # .. and of an odd number of accumulators
    (5, 32, 1, 64, 40, 128, 384),     # ranges that fit no ring of key tiles twice
])
def test_units_of_one_query_tile(layers, Hkv, heads, d, n_q, cache, chunk):
    """Up to 128 padded rows per KV head: two MMA issuers, scores written by the softmax warps."""
    path, _ = _check(layers, Hkv * heads, Hkv, d, [(n_q, 9999, chunk, cache)])
    assert path == fb.FINCH_SCORE_ONE_KERNEL


@pytest.mark.parametrize("layers,Hkv,heads,n_q,cache,chunk,group_mode,one", [
    (1, 2, 4, 129, 100, 70, 0, True),      # 544 rows: two halves of 272, three query tiles each
    (2, 2, 2, 255, 300, 300, 1, True),     # a query head each, sums over four units to a group
    (3, 2, 8, 128, 1000, 500, 0, True),    # 512 rows each
    (2, 1, 72, 8, 300, 200, 0, True),      # so many query heads that no prompt's rows are resident whole
    (1, 2, 128, 5, 100, 300, 1, True),     # .. nor more than eight of half of them
    (3, 2, 8, 129, 300, 200, 0, False),    # 544: two launches
    (1, 2, 3, 200, 300, 200, 0, False),    # an odd number of query heads
    (70, 2, 4, 160, 300, 200, 0, True),    # more halves than SMs: whole units in two windows
    (11, 8, 4, 195, 634, 1817, 0, False),  # .. whose ranges would meet across CTAs
])
def test_halves_of_a_kv_heads_queries(layers, Hkv, heads, n_q, cache, chunk, group_mode, one):
    """513 to 1024 padded rows per KV head: two units that share its keys, their column sums added."""
    path, _ = _check(layers, Hkv * heads, Hkv, 128, [(n_q, 9999, chunk, cache)], group_mode=group_mode)
    assert path == (fb.FINCH_SCORE_ONE_KERNEL if one else fb.FINCH_SCORE_TWO_LAUNCH)


@pytest.mark.parametrize("layers,heads,n_q,cache,chunk,window", [
    (3, 4, 72, 300, 66, 1),      # three query tiles, ranges of one key tile: one part of a row's statistics to a range
    (12, 4, 72, 300, 500, 2),    # .. of two
    (20, 4, 73, 500, 900, 4),    # .. of four, the last one shorter
    (3, 4, 24, 900, 200, 1),     # copies of a row, one query tile
    (3, 4, 40, 2000, 1000, 2),   # two query tiles
])
def test_parts_of_a_rows_statistics_in_short_ranges(layers, heads, n_q, cache, chunk, window):
    path, w = _check(layers, 2 * heads, 2, 128, [(n_q, 99999, chunk, cache)])
    assert (path, w) == (fb.FINCH_SCORE_ONE_KERNEL, window)
