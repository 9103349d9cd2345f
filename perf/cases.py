"""The calls that a user of this library spends time in, as cases that can be timed.

Six kinds of pass, each through the public entry points and at the sizes of the repository's workloads or generic ones:

  step     VerifyStep.run: attention of one layer, vocabulary pass, acceptance
  layer    VerifyStep.attention: one attention layer of a model's forward
  fp8      tsd_verify_attention_fp8_cache: the same layer over an 8-bit cache
  joint    one pass over the trees of two consecutive blocks: visibility, mask, attention, vocabulary pass, acceptance of
           both trees, trigger
  vocab    tsd_confidence_topk alone
  decode   BlockDecoder.decode: a few passes of the decode loop of one block, over logits a model has produced
"""
import math

import numpy as np
import torch

from paper_2608_27514_b200 import binding as B
from paper_2608_27514_b200 import workloads as W
from paper_2608_27514_b200.decode import BlockDecoder
from paper_2608_27514_b200.step import VerifyStep

DEV = "cuda:0"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------------------------------ cases
def _attn(kind, name, S, Bn, R, Nc, Hq, Hkv, d, dtype, **more):
    c = dict(kind=kind, S=S, B=Bn, R=R, Nc=Nc, Hq=Hq, Hkv=Hkv, d=d, dtype=dtype, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The reference-precision workload: fp32, four short branches, a vocabulary of 4096.  What a user runs to check a
        # model or a tree policy; the smallest whole step, where latency and launches count.
        _attn("step", "step_fp32_small", 1, 4, 32, 256, 4, 4, 64, "f32", V=4096, k=3, ragged=False),
        # One user's request: an 8-node tree over one block of an 8B-sized model (32 heads, 768 tokens of context).
        _attn("step", "step_one_request", 1, 8, 32, 736, 32, 32, 128, "bf16", V=126464, k=3, ragged=False),
        # One request with the next block speculated along (64 rows per branch), 16 branches, longer context.
        _attn("step", "step_next_block", 1, 16, 64, 1472, 32, 32, 128, "bf16", V=126464, k=3, ragged=False),
        # Batched serving: 16 sequences with full 32-node trees.
        _attn("step", "step_batch16", 16, 32, 32, 1504, 32, 32, 128, "bf16", V=126464, k=3, ragged=False),
        # Long context with grouped-query heads, 64 branches of two blocks, the wide vocabulary: the largest step.
        _attn("step", "step_long_gqa", 4, 64, 64, 5056, 28, 4, 128, "bf16", V=152064, k=4, ragged=False),
        # A small server's layer: 5 sequences of different lengths, trees cut to an odd 13 nodes, grouped heads.
        _attn("layer", "layer_ragged_gqa", 5, 13, 32, 1187, 28, 4, 128, "bf16", ragged=True),
        # The same kind of layer for a model with 64-wide heads.
        _attn("layer", "layer_head64", 4, 16, 32, 1472, 32, 8, 64, "bf16", ragged=False),
        # The cache kept as 8-bit codes so that more sequences fit: one layer of a batch of 8.
        _attn("fp8", "layer_fp8_cache", 8, 32, 32, 1504, 32, 32, 128, "bf16", ragged=True),
        # Inter-block speculation in the form of two trees per sequence, masks rebuilt for the pass.
        _attn("joint", "joint_two_trees", 2, 20, 32, 1100, 32, 8, 128, "bf16", n_next=5, V=126464, k=3, ragged=True),
        # Plain blockwise decoding, no tree: the 32 rows of one block, the wide vocabulary.
        dict(name="vocab_one_block", kind="vocab", rows=32, V=152064, k=1, dtype="bf16"),
        # fp32 logits (a model head that does not round) with a vocabulary that fits no vector width.
        dict(name="vocab_fp32_ragged", kind="vocab", rows=416, V=50257, k=5, dtype="f32"),
        # The decode loop of one block for a few requests: drafted tokens accepted by probability, longest path.
        dict(name="decode_block", kind="decode", S=3, B=10, R=32, V=126464, k=3, width=3, depth=3, passes=4, dtype="bf16",
             rule="prob", search="longest"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_any(rng):
    kind = rng.choice(["step", "step", "step", "layer", "layer", "fp8", "joint", "vocab", "vocab", "decode"])
    vocab = rng.choice([4096, 32000, 126464, 152064, 8 * _log_int(rng, 512, 19008)])
    if kind == "vocab":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        return dict(kind=kind, rows=_log_int(rng, 8, 4096), V=vocab - rng.choice([0, 0, 1, 5]), k=rng.choice([1, 2, 3, 4, 5, 8]), dtype=dtype)
    if kind == "decode":
        width, depth = rng.choice([(2, 2), (3, 2), (3, 3), (4, 3)])
        return dict(kind=kind, S=_log_int(rng, 1, 8), B=rng.randint(4, 1 + width * depth), R=32, V=vocab, k=rng.choice([3, 4]), width=width,
                    depth=depth, passes=rng.randint(2, 4), dtype="bf16", rule=rng.choice(["exact", "exact", "top1", "prob"]),
                    search=rng.choice(["greedy", "longest"]))
    if kind == "step" and rng.random() < 0.25:  # the fp32 path serves checking, at checking's sizes
        h = rng.choice([2, 4, 8])
        return _attn(kind, None, rng.choice([1, 1, 2]), rng.randint(1, 8), 32, _log_int(rng, 32, 768), h, h // rng.choice([1, 1, 2]),
                     rng.choice([64, 128]), "f32", V=8 * _log_int(rng, 128, 4096), k=rng.choice([1, 3, 4]), ragged=rng.random() < 0.3)
    group = rng.choice([1, 1, 2, 4, 7])
    hkv = rng.choice([4, 8]) if group > 1 else rng.choice([16, 32])
    d = 64 if kind == "layer" and rng.random() < 0.35 else 128
    case = _attn(kind, None, _log_int(rng, 1, 16), _log_int(rng, 1, 64), 32 if kind == "joint" else rng.choice([32, 32, 64]),
                 _log_int(rng, 64, 5056), hkv * group, hkv, d, "bf16", ragged=rng.random() < 0.5)
    if kind in ("step", "joint"):
        case.update(V=vocab, k=rng.choice([1, 3, 4]))
    if kind == "joint":
        case["B"] = max(case["B"], 5)
        case["n_next"] = rng.randint(1, 4)
    return case


def _weight(case):
    """Rough seconds of a pass at the card's rates."""
    w = work(case)
    return w["bytes"] / 6.5e12 + w["flops"] / (1.6e15 if case["dtype"] == "bf16" else 5e13)


def draw(rng):
    """A case of the ranges above: 1 to 16 sequences, 1 to 64 branches, caches of 64 to 5056 tokens, any of the head layouts,
    vocabularies of 4096 to 152064; never heavier than the largest listed one, 64-wide heads not than theirs."""
    largest = _weight(listed()[4])
    while True:
        case = _draw_any(rng)
        if _weight(case) <= 0.8 * largest and (case.get("d") != 64 or work(case)["flops"] <= 2.5e10):
            return case


# ----------------------------------------------------------------------------------------- inputs
def _config(case, seed, **more):
    kw = dict(name="case", S=case["S"], Hq=case.get("Hq", 1), Hkv=case.get("Hkv", 1), d=case.get("d", 64), Nc=case.get("Nc", 64),
              B=case["B"], R=case["R"], V=case.get("V", 4096), k=case.get("k", 1), tau=0.9, dtype=case["dtype"], sigma=3.0,
              arity=3, seed=seed)
    return W.Config(**dict(kw, **more))


def _cache_lens(case):
    """Valid cached tokens per sequence: requests of different lengths in one capacity."""
    return [case["Nc"] - (s * 7919) % (case["Nc"] // 3 + 1) if case["ragged"] else case["Nc"] for s in range(case["S"])]


def _lens_tensor(case):
    return torch.tensor(_cache_lens(case), dtype=torch.int32, device=DEV) if case["ragged"] else None


def _peaked_logits(rows, V, dtype, gen, token=None, p=None):
    """Logits of a confident head: N(0, 3^2) noise, one token per row lifted to probability p (20 % of rows above 0.9)."""
    pitch = (V + 7) // 8 * 8
    out = torch.empty((rows, pitch), dtype=dtype, device=DEV)[:, :V]
    if token is None:
        token = torch.randint(0, V - 1, (rows,), generator=gen, device=DEV)
    if p is None:
        u = torch.rand(rows, generator=gen, device=DEV)
        p = torch.where(u < 0.2, 0.93 + 0.3 * u, 0.2 + 0.7 * u)
    for r0 in range(0, rows, 1024):
        r1 = min(rows, r0 + 1024)
        x = torch.randn((r1 - r0, V), generator=gen, device=DEV).mul_(3.0)
        top = torch.logsumexp(x, 1) + torch.log(p[r0:r1] / (1 - p[r0:r1]))
        x.scatter_(1, token[r0:r1, None], top[:, None])
        out[r0:r1] = x
    return out


def _prepare_step(case, seed):
    cfg = _config(case, seed)
    step = VerifyStep.for_config(cfg, DEV)
    step.build_mask(None, _lens_tensor(case))
    vi = W.verify_inputs(cfg, DEV)
    return dict(step=step, attn=W.attention_inputs(cfg, DEV), logits=vi["logits"], parent=vi["parent"], state=vi["state"],
                mask_id=vi["mask_id"])


def _prepare_layer(case, seed):
    cfg = _config(case, seed)
    step = VerifyStep.for_config(cfg, DEV)
    step.build_mask(None, _lens_tensor(case))
    return dict(step=step, attn=W.attention_inputs(cfg, DEV))


def _prepare_fp8(case, seed):
    st = _prepare_layer(case, seed)
    a = st["attn"]
    for name in ("k", "v"):
        x = a.pop(name + "_cache").float()
        scale = x.abs().amax(dim=(1, 3)) / 448.0  # per (sequence, kv head)
        st[name + "_codes"] = (x / scale[:, None, :, None]).to(torch.float8_e4m3fn)
        st[name + "_scale"] = scale
    st["workspace"] = torch.empty(B.tsd_verify_attention_fp8_cache_workspace_bytes(st["step"].layout), dtype=torch.uint8, device=DEV)
    return st


def _prepare_joint(case, seed):
    S, Bn, R, n_next = case["S"], case["B"], case["R"], case["n_next"]
    n_cur = Bn - n_next
    cfg = _config(case, seed)
    plans = [W.plan_tree(_config(case, seed + 77 * t, B=b)) for t, b in enumerate((n_cur, n_next))]
    plan = {key: np.concatenate([p[key] for p in plans], axis=1) for key in ("state", "kind", "tok", "pstar")}
    shifted = np.where(plans[1]["parent"] < 0, -1, plans[1]["parent"] + n_cur).astype(np.int32)
    parent = np.concatenate([plans[0]["parent"], shifted], axis=1)
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device=DEV)
    return dict(step=VerifyStep.for_config(cfg, DEV), attn=W.attention_inputs(cfg, DEV), logits=W.logits_from_plan(cfg, plan, DEV),
                lens=_lens_tensor(case), n_cur=n_cur, parent=torch.from_numpy(parent).to(DEV),
                state=torch.from_numpy(plan["state"]).to(DEV), mask_id=int(plans[0]["mask_id"]),
                vis=torch.zeros((S, Bn, (Bn + 63) // 64), dtype=torch.int64, device=DEV),
                edge_valid=torch.zeros((S, Bn), dtype=torch.uint8, device=DEV), prefix_len=i32(S, Bn), node=i32(2, S), length=i32(2, S),
                gained=i32(2, S), flag=torch.zeros((2, S, R), dtype=torch.uint8, device=DEV), tok=i32(2, S, R),
                trigger=torch.zeros(S, dtype=torch.uint8, device=DEV), top_conf=torch.zeros((S, 2), device=DEV))


def _prepare_vocab(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(4000 + seed)
    n, k = case["rows"], case["k"]
    f32 = lambda *shape: torch.empty(shape, dtype=torch.float32, device=DEV)
    need = B.tsd_confidence_topk_workspace_bytes(n, case["V"], k)
    return dict(logits=_peaked_logits(n, case["V"], DTYPES[case["dtype"]], gen), k=k, conf=f32(n), prob=f32(n, k), lse=f32(n),
                idx=torch.empty((n, k), dtype=torch.int32, device=DEV), workspace=torch.zeros(max(need, 16), dtype=torch.uint8, device=DEV))


def _prepare_decode(case, seed):
    cfg = _config(case, seed)
    S, Bn, R, V = case["S"], case["B"], case["R"], case["V"]
    gen = torch.Generator(device=DEV).manual_seed(6000 + seed)
    mask_id = V - 1
    rnd = lambda *shape: torch.rand(shape, generator=gen, device=DEV)
    # a row's most likely token is the same from pass to pass, its probability drifts a little; 20 % of rows are above tau
    token = torch.randint(0, V - 1, (S, 1, R), generator=gen, device=DEV).expand(S, Bn, R).reshape(-1)
    high = (rnd(S, 1, R) < 0.2).expand(S, Bn, R).reshape(-1)
    base = rnd(S, 1, R).expand(S, Bn, R).reshape(-1)
    logits = []
    for _ in range(case["passes"]):
        p = torch.where(high, 0.93 + 0.06 * base, 0.25 + 0.5 * base) + 0.005 * rnd(S * Bn * R)
        logits.append(_peaked_logits(S * Bn * R, V, DTYPES[case["dtype"]], gen, token, p))
    root = torch.randint(0, V - 1, (S, R), generator=gen, device=DEV, dtype=torch.int32)
    masked = rnd(S, R) < 0.75
    masked[:, ::2] = True  # enough open rows that the block outlasts the passes
    root[masked] = mask_id
    rule = {"exact": B.TSD_ACCEPT_EXACT, "top1": B.TSD_ACCEPT_TOP1, "prob": B.TSD_ACCEPT_PROB}[case["rule"]]
    search = {"greedy": B.TSD_SEARCH_GREEDY, "longest": B.TSD_SEARCH_LONGEST}[case["search"]]
    step = VerifyStep.for_config(cfg, DEV)
    return dict(step=step, logits=logits, root=root, passes=case["passes"], tokens=torch.zeros((S, 512), dtype=torch.int32, device=DEV),
                start=torch.arange(S, dtype=torch.int32, device=DEV) * 32,
                decoder=BlockDecoder(step, case["width"], case["depth"], cfg.tau, mask_id, rule, search))


_PREPARE = dict(step=_prepare_step, layer=_prepare_layer, fp8=_prepare_fp8, joint=_prepare_joint, vocab=_prepare_vocab,
                decode=_prepare_decode)


def prepare(case, seed):
    return dict(_PREPARE[case["kind"]](case, int(seed) % (1 << 30)), kind=case["kind"])


# ------------------------------------------------------------------------------------------ passes
def _vocab_outputs(step):
    return dict(conf=step.conf, topk_idx=step.topk_idx, topk_prob=step.topk_prob, lse=step.lse)


def _run_step(st):
    step = st["step"]
    accepted = step.run(st["attn"], st["logits"], st["parent"], st["state"], st["mask_id"], 0.9)
    return dict(accepted, out=step.out, attn_lse=step.attn_lse, **_vocab_outputs(step))


def _run_layer(st):
    a, step = st["attn"], st["step"]
    out = step.attention(a["q"], a["k_cache"], a["v_cache"], a["k_draft"], a["v_draft"], a["sm_scale"])
    return dict(out=out, attn_lse=step.attn_lse)


def _run_fp8(st):
    a, step = st["attn"], st["step"]
    B.tsd_verify_attention_fp8_cache(step.layout, step.mask, a["q"], st["k_codes"], st["v_codes"], st["k_scale"], st["v_scale"],
                                     a["k_draft"], a["v_draft"], step.out, st["workspace"], step.attn_lse, a["sm_scale"],
                                     status=step.status)
    return dict(out=step.out, attn_lse=step.attn_lse)


def _run_joint(st):
    a, step = st["attn"], st["step"]
    B.tsd_build_interblock_vis(st["n_cur"], st["vis"])
    step.build_mask(st["vis"], st["lens"])
    out = step.attention(a["q"], a["k_cache"], a["v_cache"], a["k_draft"], a["v_draft"], a["sm_scale"])
    step.confidence_topk(st["logits"])
    B.tsd_accept_joint_trees(st["parent"], st["state"], st["n_cur"], st["mask_id"], step.conf, step.topk_idx, step.k, 0.9,
                             B.TSD_ACCEPT_EXACT, B.TSD_SEARCH_GREEDY, st["edge_valid"], st["prefix_len"], st["node"], st["length"],
                             st["gained"], st["flag"], st["tok"], step.status)
    B.tsd_interblock_trigger(st["state"], step.conf, st["node"][0], st["n_cur"], st["mask_id"], 0.9, st["trigger"], st["top_conf"],
                             step.status)
    return dict({key: st[key] for key in ("edge_valid", "prefix_len", "node", "length", "gained", "flag", "tok", "trigger", "top_conf")},
                out=out, attn_lse=step.attn_lse, **_vocab_outputs(step))


def _run_vocab(st):
    B.tsd_confidence_topk(st["logits"], st["k"], st["conf"], st["idx"], st["prob"], st["lse"], st["workspace"])
    return dict(conf=st["conf"], idx=st["idx"], prob=st["prob"], lse=st["lse"])


def _run_decode(st):
    decoder, passes = st["decoder"], iter(st["logits"])
    decoder.start(st["root"])
    root = decoder.decode(lambda state: next(passes), st["tokens"], st["start"], st["passes"])
    tree, step = decoder.tree, st["step"]
    return dict(_vocab_outputs(step), root=root, tokens=st["tokens"], fill_step=decoder.fill_step, step_base=decoder.step_base,
                n_masked=decoder.n_masked, parent=tree["parent"], state=tree["state"], node_prob=tree["prob"], n_nodes=tree["n"])


_RUN = dict(step=_run_step, layer=_run_layer, fp8=_run_fp8, joint=_run_joint, vocab=_run_vocab, decode=_run_decode)


def run(state):
    return _RUN[state["kind"]](state)


# -------------------------------------------------------------------------------------- accounting
def work(case):
    nbytes = flops = 0.0
    size = 4 if case["dtype"] == "f32" else 2
    if case["kind"] in ("step", "layer", "fp8", "joint"):
        S, N, Hq, Hkv, d = case["S"], case["B"] * case["R"], case["Hq"], case["Hkv"], case["d"]
        cached = sum(_cache_lens(case))
        nbytes += 2 * S * N * Hq * d * size + 2 * S * N * Hkv * d * size + 4 * S * N * Hq
        nbytes += 2 * cached * Hkv * d * (1 if case["kind"] == "fp8" else size)
        # every row reads the cache, its own branch and, in a joint pass, the other tree's root
        own = case["R"] * (2 if case["kind"] == "joint" else 1)
        flops += 4.0 * d * Hq * N * (cached + S * own)
    if case["kind"] in ("step", "joint", "decode"):
        rows = case["S"] * case["B"] * case["R"]
        nbytes += case.get("passes", 1) * rows * (case["V"] * size + 8 + 8 * case["k"] + 4)
    if case["kind"] == "vocab":
        nbytes += case["rows"] * (case["V"] * size + 8 + 8 * case["k"])
        rows = case["rows"]
    if case["kind"] in ("step", "joint", "decode", "vocab"):
        flops += 3.0 * case.get("passes", 1) * rows * case["V"]  # scale, exponential, sum
    return dict(bytes=nbytes, flops=flops)


def tolerance(case):
    # Four times what the outputs were seen to be off by against fp64.  bf16 attention rounds its weights and its outputs to bf16:
    # 2.3e-3 in norm, 9.3e-3 at the worst value.  Everything in fp32 (attention, probabilities, log-sum-exp): up to 3.1e-7 in norm
    # and 1.9e-6 at the worst value, from the order of sums and the last bits of exponentials; the bound leaves room for longer
    # sums than those seen.  Indices, lengths and tokens are the same.
    if case["kind"] in ("step", "layer", "fp8", "joint") and case["dtype"] == "bf16":
        return {"rel": 1e-2, "max": 4e-2, "differ": 0.0}
    return {"rel": 5e-6, "max": 2e-5, "differ": 0.0}
