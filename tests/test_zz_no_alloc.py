"""finch_score_static: the scoring call for hosts that may not allocate device memory.

Some users of the library run where cudaMalloc is not an option (a plugin inside a server whose memory pool owns
the device, a step that must not touch the driver's allocator).  They call finch_score_static, whose scratch is a
fixed array inside the library instead of a caller-supplied workspace.  These tests check that it returns what
finch_score returns, call after call, although every call reuses the same array, and that it refuses batches that
do not fit the array.  The array is 8 MiB; the tensor-core kernels need more of it than one entry per prompt row, so a
batch with few prompt rows but very many candidates stays within the row limit and still has to run on the warp-level
kernels: that case is driven on purpose, and both kinds of batch are compared with the fp64 oracle, not only with
finch_score.  The file is named to be collected last.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2408_00167_b200 import binding as fb
from paper_2408_00167_b200 import build as fbuild
from paper_2408_00167_b200 import workloads as wl
from parity_harness import ABS_TOL, REL_TOL, GpuStep, oracle_scores


@pytest.fixture(scope="module", autouse=True)
def _built():
    fbuild.build()
    fb.load()


def _case(reqs, step):
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=2, n_q_heads=8, n_kv_heads=2, head_dim=64,
                    requests=tuple(wl.Request(*r) for r in reqs), planted_frac=0.02)
    return cfg, wl.steady_state(cfg, [0, 1], step=step)


@pytest.mark.gpu
def test_static_scratch_matches_workspace_version_on_consecutive_calls():
    import torch
    # two different batches back to back: the second call finds the first call's leftovers in the shared array
    cases = [_case([(70, 9999, 150, 90), (9, 9999, 40, 33)], 2), _case([(33, 9999, 100, 260)], 3)]
    for cfg, st in cases:
        g = GpuStep(cfg, st, 2)
        try:
            fb.finch_score(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, g.scores, g.row_lse, g.ws)
            want, want_lse = g.scores.clone(), g.row_lse.clone()
            for _ in range(2):                                   # and the same batch twice in a row
                got = torch.full_like(g.scores, float("nan"))
                got_lse = torch.full_like(g.row_lse, float("nan"))
                fb.finch_score_static(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, got, got_lse)
                assert g.status() == 0
                w, x = want.cpu().numpy(), got.cpu().numpy()
                valid = ~np.isnan(w)
                assert valid.any() and np.array_equal(valid, ~np.isnan(x))
                err = np.abs(x[valid] - w[valid])
                assert np.all(err <= np.maximum(REL_TOL * np.abs(w[valid]), ABS_TOL))
                np.testing.assert_allclose(got_lse.cpu().numpy(), want_lse.cpu().numpy(), rtol=1e-5, atol=1e-5)
        finally:
            g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("reqs,tensor_cores", [
    ([(40, 10 ** 7, 700, 300)], True),          # a small batch: the tensor-core kernels fit the array
    ([(33, 10 ** 7, 140_000, 200)], False),     # 4 units x 140 200 candidates of partial sums do not: warp-level kernels
])
def test_static_scratch_on_both_kernel_paths_against_the_oracle(reqs, tensor_cores):
    import torch
    cfg, st = _case(reqs, 1)
    g = GpuStep(cfg, st, 2)
    try:
        assert fb.finch_score_static_path(g.ctx, g.batch) is tensor_cores
        ref = oracle_scores(cfg, st, threads=8)
        fb.finch_score(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, g.scores, g.row_lse, g.ws)   # always tensor cores
        want = g.scores.clone()
        for _ in range(2):
            got = torch.full_like(g.scores, float("nan"))
            fb.finch_score_static(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, got, None)
            assert g.status() == 0
            for name, x in (("static", got), ("workspace", want)):
                x = x.cpu().numpy().astype(np.float64)
                assert not np.isnan(x).any()
                bad = np.abs(x - ref) > np.maximum(REL_TOL * np.abs(ref), ABS_TOL)
                assert not bad.any(), f"{name}: {int(bad.sum())} scores outside the tolerance"
    finally:
        g.close()


def test_static_scratch_rejects_batches_beyond_its_size():
    """Host-side check, no GPU needed: a validation-only context still applies the size limit first."""
    limit = fb.finch_score_static_max_rows()
    assert limit == 1 << 20
    ctx = fb.finch_ctx_create(32, 32, 8, 64, fb.FINCH_BF16, max_batch=1, max_prompt=4096, max_candidates=8192,
                              device=-1)
    try:
        base = 0x7000_0000_0000

        def call(total_q):
            b = fb.finch_batch(1, base, base + 256, base + 512, base + 768, base + 1024, total_q, 512, 256,
                               min(total_q, 4096), 256, 512, 256)
            t = lambda slot, tok, heads: fb.finch_tensor(base + 0x1000_0000 * slot, heads * tok * 64, tok * 64, 64)
            q, ck, hk = t(1, total_q, 32), t(2, 256, 8), t(3, 512, 8)
            return fb.load().finch_score_static(ctx, C.byref(q), C.byref(ck), C.byref(hk), C.byref(b),
                                                C.c_void_p(base + 0x9000_0000), None, None)
        assert call(limit // (32 * 32)) == fb.FINCH_ERR_UNSUPPORTED            # fits: stops only at the launch
        assert call(limit // (32 * 32) + 1) == fb.FINCH_ERR_WORKSPACE_TOO_SMALL
    finally:
        fb.finch_ctx_destroy(ctx)


@pytest.mark.parametrize("L,Hkv,g,B,p,cache,chunk,tensor_cores", [
    (9, 32, 2, 1, 6, 590, 1081, True),          # a short prompt: whole query tiles of statistics for few rows
    (11, 32, 1, 1, 8, 981, 426, True),
    (64, 32, 1, 1, 8, 100, 100, True),          # more than the array holds at once: some layers at a time
    (1, 64, 1, 40, 2, 3, 1, True),              # some requests of a layer at a time
    (24, 4, 4, 16, 2, 28, 78, True),
    (32, 8, 4, 1, 128, 2048, 2048, False),      # two entries per candidate do not fit
    (32, 8, 4, 1, 205, 10, 10, False),          # 5 x 32 x 32 x 205 entries for the rows
])
def test_static_scratch_takes_the_tensor_cores_by_rows_and_candidates(L, Hkv, g, B, p, cache, chunk, tensor_cores):
    """Host arithmetic: five entries per prompt row and two per layer, KV head and candidate."""
    need = 5 * L * Hkv * g * B * p + 2 * L * Hkv * B * (cache + chunk) + B + 513
    assert (need <= fb.finch_score_static_max_rows()) is tensor_cores
    ctx = fb.finch_ctx_create(L, Hkv * g, Hkv, 64, fb.FINCH_BF16, max_batch=B, max_prompt=p, max_candidates=cache + chunk, device=-1)
    try:
        off = lambda n: [n * i for i in range(B + 1)]
        batch = fb.make_batch(off(p), off(chunk), off(cache), [cache] * B, [cache] * B, device="cpu")
        assert fb.finch_score_static_path(ctx, batch) is tensor_cores
    finally:
        fb.finch_ctx_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("L,Hkv,reqs,group_mode,self_term", [
    (65, 32, [(8, 9999, 100, 60)], 0, True),                                    # 33 + 32 layers
    (70, 32, [(5, 9999, 40, 70)], 1, False),
    (1, 64, [(1 + i % 2, 9999, 1 + i % 3, 5) for i in range(40)], 0, False),   # 20 + 20 requests
])
def test_static_scratch_in_parts_returns_what_the_workspace_call_returns(L, Hkv, reqs, group_mode, self_term):
    """Statistics that the array cannot hold at once: layers, or the requests of a layer, one part after the other."""
    import torch
    cfg = wl.scaled(wl.CONFIGS["c3"], n_layers=L, n_q_heads=Hkv, n_kv_heads=Hkv, head_dim=64, planted_frac=0.02,
                    group_mode=group_mode, requests=tuple(wl.Request(*r) for r in reqs))
    st = wl.steady_state(cfg, list(range(L)), step=1)
    lse = None
    if self_term:
        lse = np.random.default_rng(0).normal(3.0, 1.0, (L, Hkv, int(st["q_off"][-1]))).astype(np.float32)
    g = GpuStep(cfg, st, L, prompt_self_lse=lse)
    try:
        assert fb.finch_score_static_path(g.ctx, g.batch)
        fb.finch_score(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, g.scores, g.row_lse, g.ws)
        got, got_lse = torch.full_like(g.scores, float("nan")), torch.full_like(g.row_lse, float("nan"))
        before = fb.finch_launch_count(g.ctx)
        fb.finch_score_static(g.ctx, g.q, g.cache_k, g.chunk_k, g.batch, got, got_lse)
        assert g.status() == 0
        per_part = 3 + (len(reqs) > 1) + (group_mode == 1)
        assert fb.finch_launch_count(g.ctx) - before == 2 * per_part
        w, x = g.scores.cpu().numpy(), got.cpu().numpy()
        valid = ~np.isnan(w)                                    # entries behind a request's candidates stay as they were
        assert np.array_equal(valid, ~np.isnan(x))
        assert np.all(np.abs(x[valid] - w[valid]) <= np.maximum(REL_TOL * np.abs(w[valid]), ABS_TOL))
        np.testing.assert_allclose(got_lse.cpu().numpy(), g.row_lse.cpu().numpy(), rtol=1e-5, atol=1e-5)
    finally:
        g.close()
