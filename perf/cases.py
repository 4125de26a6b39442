"""The work this framework is measured on: compression steps and documents as a serving program asks for them.

A case is one of three kinds.  "step" is one finch_step (or, with `parts`, the three calls score / select / compact;
with `host`, finch_step_host) over `layers` layers of a model for `batch` requests; "document" is a whole document
through DocumentCompressor, chunk by chunk.  Inputs are seeded Gaussian or Student-t draws with planted keys that are
relevant to the prompt, the recipe of the package's own workloads, drawn on the GPU.

The kept set of a step is a discrete function of its scores: a candidate that scores within rounding of the budget's
threshold may legitimately fall on either side, and every kept row behind it then moves by one slot.  So that two
correct implementations return the same rows, `prepare` moves the few candidates that fall within MARGINS of the
threshold away from it; a document's relevant tokens stand clear of the rest by themselves, and its schedule asks for
exactly as many rows as there are relevant tokens.
"""
import math
import random

import numpy as np
import torch

from paper_2408_00167_b200 import binding as fb
from paper_2408_00167_b200 import document

MARGINS = (4e-4, 3e-4, 2e-4)   # relative distance from the threshold that `prepare` clears of candidates, in turn
ROPE_BASE = 10000.0


def _step(name=None, layers=32, q_heads=32, kv_heads=8, head_dim=128, dtype="bf16", prompt=128, cache=2048, chunk=2048,
          budget=2048, batch=1, mix=0, keys="normal", planted=0.01, groups="kv_head", rope=False, prompt_keys=False,
          causal=False, parts=False, host=False):
    """One step.  batch > 1: a ragged batch, its lengths drawn from `mix` (prompt / cache / budget are then bounds)."""
    case = dict(kind="step", layers=layers, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, dtype=dtype, prompt=prompt,
                cache=cache, chunk=chunk, budget=budget, batch=batch, mix=mix, keys=keys, planted=planted, groups=groups,
                rope=rope, prompt_keys=prompt_keys, causal=causal, parts=parts, host=host)
    return dict(case, name=name) if name else case


def _document(name=None, layers=32, q_heads=32, kv_heads=8, head_dim=128, prompt=128, tokens=32768, chunk=2048, ratio=16,
              groups="kv_head"):
    case = dict(kind="document", layers=layers, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, dtype="bf16",
                prompt=prompt, tokens=tokens, chunk=chunk, ratio=ratio, groups=groups)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call: one layer of a small fp32 model, 512 candidates, all latency
        _step("f32_one_layer", layers=1, q_heads=8, kv_heads=8, head_dim=64, dtype="f32", prompt=16, cache=256, chunk=256,
              budget=256, planted=0.03),
        # a model's forward pass hands its layers over one at a time: one layer with a short chunk ..
        _step("one_layer_1k", layers=1, cache=512, chunk=512, budget=512),
        # .. and with the full chunk of a 32K-token context
        _step("one_layer_4k", layers=1),
        # all layers at once, multi-head attention, 4096-token texts in chunks of 512
        _step("mha_1k", kv_heads=32, prompt=64, cache=512, chunk=512, budget=512, planted=0.02),
        # the headline workload: grouped-query attention, a 32K-token context in chunks of 2048
        _step("gqa_4k"),
        # a 131K-token context compressed 93 times, heavy-tailed keys
        _step("gqa_heavy_tails", prompt=64, cache=1408, budget=1408, keys="student_t3", planted=0.005),
        # sixteen requests of a serving batch, prompts of 16-256 and texts of 4K-32K tokens, 8 times compressed
        _step("ragged_batch", batch=16, mix=4, prompt=256, cache=4096, chunk=1024, budget=4096),
        # nothing a multiple of anything: an odd prompt, a short last chunk behind an odd cache
        _step("odd_sizes", layers=28, prompt=37, cache=1000, chunk=93, budget=1000),
        # the paper's own setting: one set of positions per layer (sum over all heads), the prompt's own keys in the
        # softmax, rotary keys moved to their new slots, a cache that still grows
        _step("paper_rotary", kv_heads=32, prompt=77, cache=896, chunk=512, budget=1024, groups="layer", rope=True,
              prompt_keys=True, planted=0.02),
        # the ablation that conditions on the whole input: the chunk's tokens are query rows too, and causal
        _step("condition_on_input", layers=4, prompt=128, cache=1024, chunk=1024, budget=1024, causal=True, parts=True),
        # a whole 32K-token document, the paper's growing cache
        _document("document_32k"),
        # a step whose chunk arrives in host memory, as it does when the document is encoded elsewhere
        _step("host_inputs", layers=8, host=True),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))

    q_heads, kv_heads, head_dim = rng.choice([(32, 8, 128), (32, 8, 128), (32, 32, 128), (8, 8, 64), (8, 2, 128), (16, 4, 64)])
    model = dict(layers=log(1, 32), q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim)
    prompt, chunk, cache = log(16, 256), log(64, 2048), log(256, 2048)
    grown = cache + (chunk // 4 if rng.random() < 0.3 else 0)   # the budget: the cache's length, or a growing cache
    groups = "layer" if rng.random() < 0.25 else "kv_head"
    rope, prompt_keys, keys = rng.random() < 0.25, rng.random() < 0.25, rng.choice(["normal", "normal", "student_t3"])
    kind = rng.choice(["step"] * 6 + ["f32", "ragged", "causal", "document", "host"])
    if kind == "document":
        ratio = rng.choice([4, 8, 16])
        return _document(prompt=prompt, chunk=max(chunk, 256), tokens=rng.randint(3, 8) * max(chunk, 256) - rng.randint(0, 99),
                         ratio=ratio, groups=groups, **model)
    if kind == "f32":
        return _step(dtype="f32", prompt=log(16, 64), cache=log(128, 512), chunk=log(64, 512), budget=log(128, 512), keys=keys,
                     rope=rope, **dict(model, layers=log(1, 4)))
    if kind == "ragged":
        return _step(batch=rng.randint(2, 12), mix=rng.randint(0, 10**6), prompt=log(64, 256), cache=log(512, 4096),
                     chunk=log(64, 1024), budget=4096, groups=groups, keys=keys, **model)
    if kind == "causal":
        return _step(prompt=log(16, 128), cache=cache, chunk=log(64, 1024), budget=cache, causal=True, parts=True,
                     prompt_keys=prompt_keys, **dict(model, layers=log(1, 4)))
    return _step(prompt=prompt, cache=cache, chunk=chunk, budget=grown, keys=keys, groups=groups, rope=rope,
                 prompt_keys=prompt_keys, host=kind == "host", **model)


# ---------------------------------------------------------------------------------------------- geometry

def _requests(case):
    """(prompt rows, cache rows, capacity, chunk rows, budget) of every request of a step."""
    if case["batch"] == 1:
        out = [(case["prompt"], case["cache"], max(case["cache"], case["budget"]), case["chunk"], case["budget"])]
    else:
        r = random.Random(case["mix"])
        out = []
        for _ in range(case["batch"]):
            kept = r.randint(max(64, case["cache"] // 8), case["cache"])
            out.append((r.randint(min(16, case["prompt"]), case["prompt"]), kept, kept, case["chunk"], kept))
    if case["causal"]:   # the chunk's own tokens are query rows in front of the prompt's
        out = [(p + m, c, cap, m, r) for p, c, cap, m, r in out]
    return out


def _chunks(case):
    n, m = case["tokens"], case["chunk"]
    return [min(m, n - at) for at in range(0, n, m)]


def _steps_of(case):
    """(prompt rows, cache rows, chunk rows, kept rows, visible (row, candidate) pairs) of each single-request step."""
    if case["kind"] == "document":
        c, out = 0, []
        for m in _chunks(case):
            r = c + m // case["ratio"]
            out.append((case["prompt"], c, m, r, case["prompt"] * (c + m)))
            c = r
        return out
    out = []
    for p, c, _, m, r in _requests(case):
        pairs = p * (c + m) - (m * (m - 1) // 2 if case["causal"] else 0)
        out.append((p, c, m, min(r, c + m), pairs))
    return out


def work(case):
    """Q and every candidate's K read, the kept V rows read, the kept K and V rows, positions, indices and scores
    written; one multiply-add per element of the logits."""
    e = 4 if case["dtype"] == "f32" else 2
    L, Hq, Hkv, d = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"]
    G = Hkv if case["groups"] == "kv_head" else 1
    total_bytes = flops = 0
    for p, c, m, r, pairs in _steps_of(case):
        total_bytes += L * d * e * (Hq * p + Hkv * (c + m) + Hkv * r + 2 * Hkv * r) + L * G * 4 * (c + m + 3 * r)
        flops += 2 * L * Hq * d * pairs
    return {"bytes": total_bytes, "flops": flops}


def tolerance(case):
    """Indices, positions and lengths agree exactly, copied rows bit for bit; scores are fp32 sums of exponentials of
    fp32 logits.  Re-rotated keys are rounded to bf16 once more."""
    if case.get("rope") and case["dtype"] == "bf16":
        return {"rel": 1e-3, "max": 1e-2}
    return {"rel": 1e-5}


# ---------------------------------------------------------------------------------------------- inputs

def _draws(g, shape, keys="normal"):
    x = torch.randn(shape, generator=g, device="cuda")
    if keys == "student_t3":   # normal over the root of a chi-square with three degrees of freedom over three
        chi = sum(torch.randn(shape[:-1] + (shape[-1],), generator=g, device="cuda").square_() for _ in range(3))
        x /= chi.div_(3.0).sqrt_()
    return x


def _prompt_direction(q, kv_heads):
    """Unit mean prompt query of every KV head's query heads, [Hkv][d]; q is one layer's [Hq][rows][d]."""
    mean = q.float().reshape(kv_heads, -1, q.shape[-1]).mean(1)
    return mean / mean.norm(dim=-1, keepdim=True)


def _plant(g, k, direction, count, least=2.0):
    """k [Hkv][n][d] += beta sqrt(d) direction at `count` positions, beta uniform in least..4 per head."""
    if count:
        at = torch.randperm(k.shape[1], generator=g, device="cuda")[:count]
        beta = least + (4.0 - least) * torch.rand((k.shape[0], 1, 1), generator=g, device="cuda")
        k[:, at] += beta * math.sqrt(k.shape[-1]) * direction[:, None, :]


def _scores(q, k, groups, self_lse, limit):
    """The step's scores of one layer and request, [groups][N]: q [Hq][rows][d], k [Hkv][N][d]."""
    g = q.shape[0] // k.shape[0]
    total = []
    for h in range(k.shape[0]):
        s = torch.matmul(q[h * g:(h + 1) * g].float(), k[h].float().T) / math.sqrt(q.shape[-1])
        if limit is not None:
            s.masked_fill_(torch.arange(s.shape[-1], device=s.device)[None, None, :] >= limit[None, :, None], -math.inf)
        lse = torch.logsumexp(s, dim=-1)
        if self_lse is not None:
            lse = torch.logaddexp(lse, self_lse[h * g:(h + 1) * g])
        w = torch.exp_(s.sub_(lse[..., None]))
        if limit is not None:   # per-row normalisation: the fraction of the candidates a row sees
            w *= (limit / s.shape[-1])[None, :, None]
        total.append(w.sum((0, 1)))
    total = torch.stack(total)
    return total if groups == total.shape[0] else total.sum(0, keepdim=True)


def _settle(q, k, groups, r, self_lse, limit):
    """Clear the budget's threshold: the keys of candidates that score close to it are lengthened (if they are in the
    kept set) or shortened (if not) by a thirty-second, which moves their scores by a few per cent.  The others' scores
    move a little with them, hence the rounds."""
    n = k.shape[1]
    if r >= n:
        return k
    rank = torch.arange(n, device=k.device)
    for margin in MARGINS:
        s = _scores(q, k, groups, self_lse, limit)
        value, order = s.sort(dim=1, descending=True, stable=True)
        middle = (value[:, r - 1] + value[:, r]) * 0.5
        near = (value - middle[:, None]).abs() < margin * middle[:, None]
        gain = torch.where(near, torch.where(rank < r, 1 + 1 / 32, 1 - 1 / 32), torch.ones_like(value))
        gain = torch.empty_like(s).scatter_(1, order, gain).repeat_interleave(k.shape[0] // groups, 0)
        k = (k.float() * gain[..., None]).to(k.dtype)
    return k


class _State:
    """A program's buffers, batch description and context; the context is freed with it."""
    ctx = doc = None

    def __del__(self):
        torch.cuda.synchronize()
        if self.doc:
            self.doc.close()
        fb.finch_ctx_destroy(self.ctx)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 17)
    return _prepare_document(case, g) if case["kind"] == "document" else _prepare_step(case, g)


def _prepare_step(case, g):
    s = _State()
    s.case = case
    L, Hq, Hkv, d = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"]
    G = Hkv if case["groups"] == "kv_head" else 1
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    reqs = _requests(case)
    B = len(reqs)
    q_off, cache_off, chunk_off = (np.concatenate([[0], np.cumsum([r[i] for r in reqs])]).astype(np.int32) for i in (0, 2, 3))
    total_q, total_cache, total_chunk = int(q_off[-1]), int(cache_off[-1]), int(chunk_off[-1])

    def rows(heads, tokens):
        return torch.zeros((L, heads, tokens, d), dtype=dtype, device="cuda")

    s.q, s.cache_k, s.cache_v = rows(Hq, total_q), rows(Hkv, total_cache), rows(Hkv, total_cache)
    s.chunk_k, s.chunk_v = rows(Hkv, total_chunk), rows(Hkv, total_chunk)
    s.cache_pos = torch.zeros((L, G, total_cache), dtype=torch.int32, device="cuda")
    self_lse = limit = None
    if case["prompt_keys"]:   # log-sum-exp over the causally visible prompt keys, about log(row) + 1/2
        prompt_rows = torch.cat([torch.arange(1, r[0] + 1) for r in reqs]).float().cuda()
        self_lse = torch.log(prompt_rows) + 0.5 + 0.3 * torch.randn((L, Hq, total_q), generator=g, device="cuda")
    if case["causal"]:        # chunk token i sees the cache and the chunk up to itself, the prompt sees everything
        limit = torch.cat([torch.cat([torch.arange(c + 1, c + m + 1), torch.full((p - m,), c + m)])
                           for p, c, _, m, _ in reqs]).to(torch.int32).cuda()
    for b, (p, c, cap, m, r) in enumerate(reqs):
        qs = slice(int(q_off[b]), int(q_off[b]) + p)
        cs = slice(int(cache_off[b]), int(cache_off[b]) + c)
        hs = slice(int(chunk_off[b]), int(chunk_off[b]) + m)
        # the kept positions of earlier chunks: an increasing sample, one for each layer and group
        s.cache_pos[:, :, cs] = torch.rand((L, G, c), generator=g, device="cuda").add_(0.01).cumsum(-1).mul_(8).int()
        for l in range(L):
            q = _draws(g, (Hq, p, d)).to(dtype)
            k = _draws(g, (Hkv, c + m, d), case["keys"])
            _plant(g, k, _prompt_direction(q, Hkv), round(case["planted"] * (c + m)))
            k = _settle(q, k.to(dtype), G, r, None if self_lse is None else self_lse[l, :, qs], None if limit is None else limit[qs])
            v = _draws(g, (Hkv, c + m, d), case["keys"]).to(dtype)
            s.q[l, :, qs] = q
            s.cache_k[l, :, cs], s.chunk_k[l, :, hs] = k[:, :c], k[:, c:]
            s.cache_v[l, :, cs], s.chunk_v[l, :, hs] = v[:, :c], v[:, c:]
    s.chunk_pos = torch.cat([torch.arange(16 * c, 16 * c + m) for _, c, _, m, _ in reqs]).to(torch.int32).cuda()
    s.out_k, s.out_v = torch.zeros_like(s.cache_k), torch.zeros_like(s.cache_v)
    s.out_pos, s.kept_idx = torch.zeros_like(s.cache_pos), torch.zeros_like(s.cache_pos)
    s.out_len = torch.zeros(B, dtype=torch.int32, device="cuda")
    s.scores = torch.zeros((L, G, total_cache + total_chunk), dtype=torch.float32, device="cuda")
    s.row_lse = torch.zeros((L, Hq, total_q), dtype=torch.float32, device="cuda") if case["parts"] else None
    s.batch = fb.make_batch(q_off, chunk_off, cache_off, [r[1] for r in reqs], [r[4] for r in reqs],
                            prompt_self_lse=self_lse, row_limit=limit, row_norm=case["causal"])
    s.ctx = fb.finch_ctx_create(L, Hq, Hkv, d, fb.FINCH_F32 if case["dtype"] == "f32" else fb.FINCH_BF16,
                                fb.FINCH_GROUP_PER_KV_HEAD if case["groups"] == "kv_head" else fb.FINCH_GROUP_PER_LAYER,
                                max_batch=B, max_prompt=max(r[0] for r in reqs), max_candidates=max(r[1] + r[3] for r in reqs),
                                rope_theta=ROPE_BASE if case["rope"] else 0.0)
    s.ws = torch.empty(fb.finch_workspace_bytes(s.ctx, s.batch), dtype=torch.uint8, device="cuda")
    if case["host"]:          # this step's inputs wait in pinned host memory, the tensors above receive them
        s.host_q, s.host_k, s.host_v, s.host_pos = (t.cpu().pin_memory() for t in (s.q, s.chunk_k, s.chunk_v, s.chunk_pos))
        s.host_kept, s.host_len = s.kept_idx.cpu().pin_memory(), s.out_len.cpu().pin_memory()
    torch.cuda.synchronize()
    return s


def _prepare_document(case, g):
    s = _State()
    s.case = case
    L, Hq, Hkv, d = case["layers"], case["q_heads"], case["kv_heads"], case["head_dim"]
    chunks, ratio = _chunks(case), case["ratio"]
    k_target = sum(m // ratio for m in chunks)
    s.budgets = document.paper_budgets(chunks, ratio, k_target)
    s.q = torch.zeros((L, Hq, case["prompt"], d), dtype=torch.bfloat16, device="cuda")
    s.chunks = []
    for l in range(L):        # the prompt's rows share a direction of their KV head
        lead = torch.nn.functional.normalize(torch.randn((Hkv, 1, 1, d), generator=g, device="cuda"), dim=-1)
        s.q[l] = (_draws(g, (Hkv, Hq // Hkv, case["prompt"], d)) + 6.0 * lead).reshape(Hq, case["prompt"], d)
    for i, m in enumerate(chunks):
        k, v = (torch.empty((L, Hkv, m, d), dtype=torch.bfloat16, device="cuda") for _ in range(2))
        for l in range(L):    # one token in `ratio` is relevant to the prompt, elsewhere in every layer
            kl = _draws(g, (Hkv, m, d))
            _plant(g, kl, _prompt_direction(s.q[l], Hkv), m // ratio, least=3.0)
            k[l], v[l] = kl, _draws(g, (Hkv, m, d))
        pos = torch.arange(i * case["chunk"], i * case["chunk"] + m, dtype=torch.int32, device="cuda")
        s.chunks.append((k, v, pos, m))
    s.doc = document.DocumentCompressor(
        L, Hq, Hkv, d, fb.FINCH_BF16, [k_target], max_prompt=case["prompt"], max_chunk=max(chunks),
        group_mode=fb.FINCH_GROUP_PER_KV_HEAD if case["groups"] == "kv_head" else fb.FINCH_GROUP_PER_LAYER)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------------------------- one pass

def run(s):
    case = s.case
    if case["kind"] == "document":
        s.doc.reset()
        for (k, v, pos, m), budget in zip(s.chunks, s.budgets):
            s.doc.step(s.q, [0, case["prompt"]], k, v, pos, [0, m], [budget])
        return {"k": s.doc.cache_k, "v": s.doc.cache_v, "pos": s.doc.cache_pos, "kept": s.doc.kept_idx}
    out = {"k": s.out_k, "v": s.out_v, "pos": s.out_pos, "kept": s.kept_idx, "len": s.out_len}
    if case["host"]:
        fb.finch_step_host(s.ctx, s.host_q, s.host_k, s.host_v, s.host_pos, s.q, s.chunk_k, s.chunk_v, s.chunk_pos, s.cache_k,
                           s.cache_v, s.cache_pos, s.batch, s.out_k, s.out_v, s.out_pos, s.kept_idx, s.out_len, s.host_kept,
                           s.host_len, s.ws)
        return dict(out, host_kept=s.host_kept, host_len=s.host_len)
    if case["parts"]:
        fb.finch_score(s.ctx, s.q, s.cache_k, s.chunk_k, s.batch, s.scores, s.row_lse, s.ws)
        fb.finch_select(s.ctx, s.scores, s.batch, s.kept_idx, s.out_len)
        fb.finch_compact(s.ctx, s.kept_idx, s.out_len, s.cache_k, s.cache_v, s.cache_pos, s.chunk_k, s.chunk_v, s.chunk_pos,
                         s.batch, s.out_k, s.out_v, s.out_pos)
        return dict(out, scores=s.scores, row_lse=s.row_lse)
    fb.finch_step(s.ctx, s.q, s.cache_k, s.cache_v, s.cache_pos, s.chunk_k, s.chunk_v, s.chunk_pos, s.batch, s.out_k, s.out_v,
                  s.out_pos, s.kept_idx, s.out_len, s.scores, s.ws)
    return dict(out, scores=s.scores)
