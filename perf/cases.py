"""Measured workloads of the speculative-decoding attention path.

A case is a dict of plain values.  ``listed()`` holds the fixed ones, ``draw(rng)`` gives another of
the same ranges.  ``prepare`` makes what a serving program has in hand before a call (the resident KV
cache, queries, output buffers, workspaces and, where the launches are captured, the graph), ``run``
makes one pass through the public entry points, ``work`` counts the bytes and operations a pass cannot
do without and ``tolerance`` states how far two correct implementations may lie apart.

Kinds of pass:
  round    one speculation round of the attention side through ``runner.SpecStepRunner``: verification
           of k + 1 rows layer by layer, index rebuild of all layers, k drafting steps layer by layer
  verify   the verification calls of ``layers`` consecutive layers
  select   the index rebuild of all layers in one call
  draft    k drafting steps, layer by layer, captured into a graph as a decoder would replay them
  accept   greedy prefix acceptance over the target's logits plus the drafted tokens' entropies
  control  the scalar tail of one sequence's round: argmax with entropy of the drafted rows, the
           controller's update and length selection, the length bookkeeping
"""
from __future__ import annotations

import dataclasses

import torch

from paper_2607_27735_b200 import binding, inputs
from paper_2607_27735_b200.runner import SpecStepRunner

# Shapes (query heads, KV heads, head_dim) that the repository's configurations and tests use.
_TINY, _G4, _G5 = (8, 2, 64), (32, 8, 128), (40, 8, 128)


def _attn(name, kind, shape, layers, ctx, k, budget, sink=4, recent=64, page=0, dist="normal", queries="direction",
          planted=0.01, kv="bf16", per_head=False, bf16_out=False, lse=False, graph=True):
    hq, hkv, d = shape
    case = dict(kind=kind, layers=layers, q_heads=hq, kv_heads=hkv, dim=d, ctx=",".join(str(t) for t in ctx), k=k,
                budget=budget, sink=sink, recent=recent, page=page, dist=dist, queries=queries, planted=planted, kv=kv,
                per_head=per_head, bf16_out=bf16_out, lse=lse, graph=graph)
    return dict(case, name=name) if name else case


def listed():
    return [
        # The smallest use: one tiny layer at 2 K context called straight from Python, every launch paid.
        _attn("round_tiny_eager", "round", _TINY, 1, [2048], 4, 256, planted=8, graph=False),
        # The headline: one long-context sequence of the 8B attention shape, all 32 layers, captured.
        _attn("round_8b_32k", "round", _G4, 32, [32768], 8, 2048),
        # Ordinary serving: sixteen short and middling conversations of odd lengths on 64-token pages.
        _attn("round_chat_batch16", "round", _G4, 4, [611, 5333, 1027, 2890, 745, 3999, 1500, 6143, 912, 2049, 4750, 1333,
                                                     3217, 680, 5801, 1111], 4, 512, page=64),
        # Very long context with a long speculation window: the most query rows per key.
        _attn("verify_8b_128k_k16", "verify", _G4, 1, [131072], 16, 4096, planted=0.005),
        # A ragged batch on shuffled 16-token pages, flat scores.
        _attn("verify_ragged_paged", "verify", _G4, 1, [44631, 9107, 60212, 21940, 35555, 65529, 14003, 50876], 6, 1024,
              page=16, queries="iid", planted=0),
        # The 32B shape, groups of five, heavy-tailed cache, bf16 output for the projection and the row LSE.
        _attn("verify_32b_64k", "verify", _G5, 1, [65536] * 4, 6, 2048, 8, 256, dist="student_t3", bf16_out=True, lse=True),
        # Half the cache memory: e4m3 bytes with scales, layer after layer.
        _attn("verify_8b_32k_fp8", "verify", _G4, 4, [32768], 8, 2048, kv="fp8"),
        # Index rebuild of all layers behind a 128 K context (length not a multiple of anything).
        _attn("select_8b_128k", "select", _G4, 32, [131021], 8, 4096),
        # Drafting of the 32B shape at batch 4.
        _attn("draft_32b_64k", "draft", _G5, 4, [65536] * 4, 6, 2048, 8, 256),
        # Drafting of a ragged batch over the 8-bit cache.
        _attn("draft_ragged_fp8", "draft", _G4, 2, [44631, 9107, 60212, 21940, 35555, 65529, 14003, 50876], 6, 1024, page=16,
              queries="iid", kv="fp8", bf16_out=True),
        # Acceptance for 64 sequences and the entropies of their drafted tokens, 128256-entry vocabulary.
        dict(name="accept_batch64", kind="accept", batch=64, k=8, vocab=128256, dtype="bf16"),
        # The scalar tail of one sequence's round, called from Python between two steps.
        dict(name="control_k8", kind="control", batch=1, k=8, vocab=128256, dtype="bf16"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["round", "round", "verify", "verify", "verify", "select", "draft", "draft", "accept", "control"])
    if kind in ("accept", "control"):
        vocab = rng.choice([32000, 50257, 128256, 151936])
        dtype = rng.choice(["bf16", "bf16", "fp32"])
        batch = 1 if kind == "control" else _log_uniform(rng, 1, 96)
        return dict(kind=kind, batch=batch, k=rng.randint(1, 16 if kind == "control" else 8), vocab=vocab, dtype=dtype)
    shape = rng.choice([_G4, _G4, _G4, _G5, (24, 8, 128), (16, 2, 128), (8, 8, 128), _TINY])
    hq, hkv, d = shape
    group = hq // hkv
    page = rng.choice([0, 0, 16, 64])
    kv = rng.choice(["bf16", "bf16", "fp8"]) if d == 128 and kind in ("verify", "draft") else "bf16"
    k = rng.choice([1, 2, 3, 4, 5, 6, 7, 8, 8, 16])
    while (k + 1) * group > 128:
        k -= 1
    # tokens over all sequences and layers: at most what the largest listed case reads, spread over its logarithm
    tokens = _log_uniform(rng, 1500, 300000)
    batch = _log_uniform(rng, 1, max(1, min(16, tokens // 700)))
    ctx = []
    for _ in range(batch):
        ctx.append(max(300, min(131072, int(tokens / batch * rng.uniform(0.4, 1.6)))))
    layers = max(1, min(8, 600000 // sum(ctx), _log_uniform(rng, 1, 8)))
    budget = rng.choice([256, 512, 1000, 1024, 2048, 4096])
    budget = max(192, min(budget, max(ctx) // 2))
    return _attn(None, kind, shape, layers, ctx, k, budget, page=page, dist=rng.choice(["normal", "student_t3"]),
                 queries="iid" if kind in ("verify", "draft") and rng.random() < 0.3 else "direction",
                 kv=kv, per_head=kind == "round" and rng.random() < 0.2,
                 bf16_out=kind in ("verify", "draft") and rng.random() < 0.5,
                 lse=kind == "verify" and rng.random() < 0.5, graph=kind != "round" or rng.random() < 0.7)


# ---------------------------------------------------------------------------------------------


def _ctx(case):
    return [int(t) for t in case["ctx"].split(",")]


def _sets(case):
    return case["q_heads"] if case["per_head"] else case["kv_heads"]


def _make(case, seed, device="cuda"):
    """The seeded cache and queries of an attention case (``inputs.make_case``)."""
    ctx = _ctx(case)
    iid = case["queries"] == "iid"
    cfg = inputs.SpecConfig(
        case.get("name", "drawn"), case["layers"], len(ctx), case["q_heads"], case["kv_heads"], case["dim"],
        (min(ctx), max(ctx)), case["k"] + 1, case["budget"], case["sink"], case["recent"], case["k"],
        page_size=case["page"], shuffled_pages=case["page"] > 0, planted=0 if iid else case["planted"],
        planted_mult=3.0, planted_noise=True, kv_dist=case["dist"], q_mode="iid" if iid else "direction",
        q_std=case["dim"] ** -0.5, seed=seed % 1000003)
    made = inputs.make_case(cfg, device=device, ctx_override=ctx)
    if case["kv"] == "fp8":
        made = dataclasses.replace(made, kv=inputs.quantize_kv_fp8(made.kv))
    return made


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed * 7919 + 13)


def prepare(case, seed):
    return {"round": _prepare_round, "verify": _prepare_verify, "select": _prepare_select, "draft": _prepare_draft,
            "accept": _prepare_logits, "control": _prepare_logits}[case["kind"]](case, seed)


def run(state):
    return state["run"](state)


def _prepare_round(case, seed):
    r = SpecStepRunner(_make(case, seed), per_head=case["per_head"])
    if case["graph"]:
        r.capture()
    return dict(run=_run_round, runner=r)


def _run_round(s):
    r = s["runner"]
    r.replay() if r.graphs is not None else r.step()
    return dict(out_v=r.out_v, stats=r.stats, indices=r.indices, n=r.n_idx, out_d=r.out_d)


def _prepare_verify(case, seed):
    c = _make(case, seed)
    kv, cfg = c.kv, c.cfg
    L, B, dev = kv.n_layers, kv.batch, kv.k.device
    layers = [kv.layer_slice(l, l + 1) for l in range(L)]
    max_ctx = max(_ctx(case))
    return dict(
        run=_run_verify, layers=layers, q=[c.q_verify[l:l + 1] for l in range(L)], ctx_len=c.ctx_len, max_ctx=max_ctx,
        bf16_out=case["bf16_out"],
        out=torch.empty(L, B, cfg.n_q, kv.n_q_heads, kv.head_dim, device=dev,
                        dtype=torch.bfloat16 if case["bf16_out"] else torch.float32),
        lse=torch.empty(L, B, cfg.n_q, kv.n_q_heads, device=dev) if case["lse"] else None,
        stats=torch.zeros(L, B, kv.n_kv_heads, (max_ctx + 127) // 128 * 128, device=dev),
        ws=binding.alloc_workspace(binding.workspace_bytes(binding.WS_VERIFY, layers[0], cfg.n_q, max_ctx), dev))


def _run_verify(s):
    for l, kv in enumerate(s["layers"]):
        binding.spec_verify_attn(kv, s["q"][l], s["ctx_len"], s["max_ctx"], out=s["out"][l:l + 1],
                                 lse=None if s["lse"] is None else s["lse"][l:l + 1], stats=s["stats"][l:l + 1],
                                 workspace=s["ws"], want_lse=s["lse"] is not None, out_bf16=s["bf16_out"])
    return dict(out=s["out"], stats=s["stats"], lse=s["lse"])


def _prepare_select(case, seed):
    # scores as the verification leaves them: sums of softmax probabilities, log-normal over the background
    # with a small share of heavy hitters far above it
    ctx, L, H = _ctx(case), case["layers"], case["kv_heads"]
    gen = _generator(seed)
    T, B = max(ctx), len(ctx)
    stats = torch.zeros(L, B, H, (T + 127) // 128 * 128, device="cuda")
    rows = (case["k"] + 1) * case["q_heads"] // H
    for l in range(L):
        x = torch.randn(B, H, T, generator=gen, device="cuda").mul_(0.6).exp_()
        x.mul_(torch.where(torch.rand(B, H, T, generator=gen, device="cuda") < max(case["planted"], 1e-4), 400.0, 1.0))
        for b in range(B):
            x[b, :, ctx[b]:] = 0.0
        stats[l, :, :, :T] = x * (rows / x.sum(-1, keepdim=True))
    return dict(run=_run_select, case=case, stats=stats, sel_len=torch.tensor(ctx, dtype=torch.int32, device="cuda"),
                indices=torch.empty(L, B, H, case["budget"], dtype=torch.int32, device="cuda"),
                n=torch.empty(L, B, H, dtype=torch.int32, device="cuda"))


def _run_select(s):
    c = s["case"]
    binding.spec_select_recall(s["stats"], s["sel_len"], c["sink"], c["recent"], c["budget"], indices=s["indices"],
                               n_indices=s["n"])
    return dict(indices=s["indices"], n=s["n"])


def _prepare_draft(case, seed):
    c = _make(case, seed)
    kv, cfg = c.kv, c.cfg
    L, B, S, k, dev = kv.n_layers, kv.batch, _sets(case), case["k"], kv.k.device
    gen = _generator(seed)
    indices = torch.full((L, B, S, cfg.k_total), -1, dtype=torch.int32, device=dev)
    n = torch.empty(L, B, S, dtype=torch.int32, device=dev)
    for b, T in enumerate(_ctx(case)):
        keep = min(T, cfg.k_total)
        score = torch.rand(L, S, T, generator=gen, device=dev)
        score[:, :, :cfg.k_sink] = 2.0  # sink and recent tokens are always kept
        score[:, :, T - cfg.k_recent:] = 2.0
        indices[:, b, :, :keep] = score.topk(keep, dim=-1).indices.sort(dim=-1).values.int()
        n[:, b] = keep
    s = dict(
        run=_run_draft, layers=[kv.layer_slice(l, l + 1) for l in range(L)], bf16_out=case["bf16_out"], k=k,
        q=c.q_draft, idx=[indices[l:l + 1] for l in range(L)], n=[n[l:l + 1] for l in range(L)],
        tail_start=c.ctx_len.clone(), cur=[(c.ctx_len + j + 1).contiguous() for j in range(k)],
        out=torch.empty(k, L, B, kv.n_q_heads, kv.head_dim, device=dev,
                        dtype=torch.bfloat16 if case["bf16_out"] else torch.float32),
        ws=binding.alloc_workspace(binding.workspace_bytes(binding.WS_DRAFT, kv.layer_slice(0, 1), k_total=cfg.k_total + k),
                                   dev))
    _draft_calls(s)  # warm-up outside the capture
    torch.cuda.synchronize()
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["graph"]):
        _draft_calls(s)
    return s


def _draft_calls(s):
    for j in range(s["k"]):
        for l, kv in enumerate(s["layers"]):
            # index sets and lengths stand since before the round: every call but the first may gather early
            binding.spec_sparse_draft_attn(kv, s["q"][j, l:l + 1], s["idx"][l], s["n"][l], s["tail_start"], s["cur"][j],
                                           s["k"], out=s["out"][j, l:l + 1], workspace=s["ws"], want_lse=False,
                                           out_bf16=s["bf16_out"], early_gather=j + l > 0)


def _run_draft(s):
    s["graph"].replay()
    return s["out"]


def _prepare_logits(case, seed):
    # a language model's next-token logits: a background whose spread differs from row to row and a few
    # boosted tokens; drafted tokens that agree with the target for the first few positions
    gen = _generator(seed)
    B, k, V = case["batch"], case["k"], case["vocab"]
    rows = B * (k + 1)
    spread = torch.rand(rows, 1, generator=gen, device="cuda") * 3.8 + 0.2
    x = torch.randn(rows, V, generator=gen, device="cuda") * spread
    cols = torch.randint(0, V, (rows, 4), generator=gen, device="cuda")
    x.scatter_add_(1, cols, torch.rand(rows, 4, generator=gen, device="cuda") * 14.0)
    logits = x.to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32).view(B, k + 1, V)
    draft = logits[:, :k].argmax(-1).int()
    wrong = torch.rand(B, k, generator=gen, device="cuda") < 0.25
    draft = torch.where(wrong, (draft + 1) % V, draft).int().contiguous()
    i32 = dict(dtype=torch.int32, device="cuda")
    s = dict(run=_run_accept if case["kind"] == "accept" else _run_control, logits=logits, draft=draft, k=k,
             target=torch.empty(B, k + 1, **i32), n_accepted=torch.empty(B, **i32), next_token=torch.empty(B, **i32),
             rows=logits.view(rows, V), entropy=torch.empty(rows, device="cuda"))
    if case["kind"] == "control":
        s.update(token=torch.empty(k, **i32), entropy=torch.empty(k, device="cuda"), rows=logits[0, :k],
                 m=torch.randint(0, k + 1, (1,), generator=gen, **i32), start=torch.tensor([1.0, 4.0], device="cuda"),
                 state=torch.empty(2, device="cuda"), cand=torch.arange(1, k + 1, **i32), k_star=torch.empty(1, **i32),
                 p=torch.empty(k, device="cuda"), score=torch.empty(k, device="cuda"),
                 first=torch.tensor([5000 + seed % 1000], **i32), committed=torch.empty(1, **i32),
                 ctx_verify=torch.empty(1, **i32), cur_len=torch.empty(k, 1, **i32))
    return s


def _run_accept(s):
    binding.spec_accept_greedy(s["logits"], s["draft"], target=s["target"], n_accepted=s["n_accepted"],
                               next_token=s["next_token"])
    binding.spec_token_entropy(s["rows"], entropy=s["entropy"])
    return dict(target=s["target"], n_accepted=s["n_accepted"], next_token=s["next_token"], entropy=s["entropy"])


def _run_control(s):
    s["state"].copy_(s["start"])  # the tracked means and the length as the previous round left them
    s["committed"].copy_(s["first"])
    binding.spec_token_argmax(s["rows"], token=s["token"], entropy=s["entropy"])
    binding.spec_controller_update(s["state"], s["entropy"], s["m"], 0.9)
    binding.spec_controller_select(s["state"], s["entropy"], s["cand"], 0.05, 1.0, k_star=s["k_star"], p=s["p"],
                                   score=s["score"])
    binding.spec_advance_lengths(s["committed"], s["m"], s["k"], s["ctx_verify"], s["cur_len"])
    return {n: s[n] for n in ("token", "entropy", "state", "k_star", "p", "score", "committed", "ctx_verify", "cur_len")}


# ---------------------------------------------------------------------------------------------


def work(case):
    if case["kind"] in ("accept", "control"):
        es = 2 if case["dtype"] == "bf16" else 4
        rows = case["batch"] * (case["k"] + 1) if case["kind"] == "accept" else case["k"]
        return {"bytes": rows * case["vocab"] * es + 8 * rows, "flops": 4.0 * rows * case["vocab"]}
    ctx, L, D, Hq, Hkv, k = _ctx(case), case["layers"], case["dim"], case["q_heads"], case["kv_heads"], case["k"]
    es, oes, sets = (1 if case["kv"] == "fp8" else 2), (2 if case["bf16_out"] else 4), _sets(case)
    tokens = sum(ctx)
    n_bytes = flops = 0.0
    if case["kind"] in ("round", "verify"):
        n_bytes += L * (tokens * Hkv * D * 2 * es + tokens * sets * 4 + len(ctx) * (k + 1) * Hq * D * (2 + oes))
        flops += 4.0 * L * tokens * Hq * (k + 1) * D
    if case["kind"] in ("round", "select"):
        n_bytes += L * sets * 4 * (tokens + len(ctx) * case["budget"])
    if case["kind"] in ("round", "draft"):
        for j in range(k):
            rows = sum(min(case["budget"], t) + j + 1 for t in ctx)
            n_bytes += L * (rows * sets * (D * 2 * es + 4) + len(ctx) * Hq * D * (2 + oes))
            flops += 4.0 * L * rows * Hq * D
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "select":
        return "exact"
    if kind in ("accept", "control"):
        # tokens and lengths are whole numbers; entropies and scores are fp32 sums over the vocabulary with
        # hardware exponentials
        return {"rel": 1e-4, "max": 1e-3, "differ": 0.0}
    if kind == "round":
        # Two keys whose scores agree to the last bits of an fp32 sum may change places at the edge of the
        # budget: about one in four hundred index sets.  Such a set is shifted by one between the two keys,
        # and its drafting sees one other key of some thousand.
        return {"rel": 2e-3, "max": 0.5, "differ": 0.01}
    # fp32 results of bf16 (or exactly expanded e4m3) operands: fp32 accumulation, probabilities carried in
    # two 16-bit terms, hardware exponentials; or the same rounded to bf16
    return {"rel": 1e-2 if case["bf16_out"] else 1e-4}
