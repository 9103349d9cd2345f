"""The step in one call (attention beside the vocabulary pass) against the three calls it stands for."""
import subprocess
import sys

import pytest
import torch

from paper_2608_27514_b200 import workloads as W
from paper_2608_27514_b200.step import VerifyStep

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("kw", [dict(Hq=2, Hkv=2, V=4096), dict(Hq=32, Hkv=8, B=1, Nc=64, V=152064), dict(S=3, B=9, Hq=8, Hkv=4, Nc=1000, V=32000),
                                dict(B=64, V=126464), dict(d=64, Hq=4, Hkv=4, V=126464), dict(dtype="f32", d=64, Hq=4, Hkv=4, Nc=100, V=4096)])
def test_step_in_one_call_equals_the_three_calls(kw):
    # few and many rows against few and many attention items; the logits are rewritten in place before every pass, so that a
    # pass that ran ahead of its inputs, or read what an SM had kept of the old ones, would show; every result bit for bit
    cfg = W.small(W.CONFIGS["cfg2"], name="case", **kw)
    attn, vi = W.attention_inputs(cfg, DEV), W.verify_inputs(cfg, DEV)
    one, three = VerifyStep.for_config(cfg, DEV), VerifyStep.for_config(cfg, DEV)
    logits = vi["logits"]
    for i in range(8):
        logits = torch.roll(logits, 1 + 37 * i, 1)
        vi["logits"].copy_(logits)
        attn["q"].mul_(-1.0)
        a = one.run(attn, vi["logits"], vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
        after = one.out.clone(), one.attn_lse.clone(), one.conf.clone()
        three.attention(attn["q"], attn["k_cache"], attn["v_cache"], attn["k_draft"], attn["v_draft"], attn["sm_scale"])
        three.confidence_topk(vi["logits"])
        b = three.accept(vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
        assert torch.equal(after[0], three.out) and torch.equal(after[1], three.attn_lse) and torch.equal(after[2], three.conf)
        for x, y in ((one.topk_idx, three.topk_idx), (one.topk_prob, three.topk_prob), (one.lse, three.lse)):
            assert torch.equal(x, y)
        for key in a:
            assert torch.equal(a[key], b[key]), key
    one.check_status()


@pytest.mark.parametrize("kw", [dict(B=2, Nc=300, Hq=32, Hkv=8, V=32000), dict(B=2, Nc=5056, Hq=4, Hkv=2, V=126464),
                                dict(B=1, Nc=1500, Hq=28, Hkv=4, V=152064), dict(B=2, Nc=700, Hq=28, Hkv=4, V=50008, d=64),
                                dict(dtype="f32", B=3, d=128, Hq=4, Hkv=2, Nc=100, V=5004), dict(dtype="f32", B=4, d=64, Hq=4, Hkv=4, Nc=100, V=32768)])
def test_step_with_the_vocabulary_pass_beside_the_attention(kw):
    # both orders of the two kernels, whole items and items shared by a cluster; a kernel of the caller's right behind the step
    # sees both results, and the next step may follow at once on the same buffers
    test_step_in_one_call_equals_the_three_calls(kw)
    cfg = W.small(W.CONFIGS["cfg2"], name="case", **kw)
    attn, vi = W.attention_inputs(cfg, DEV), W.verify_inputs(cfg, DEV)
    step = VerifyStep.for_config(cfg, DEV)
    seen = []
    for _ in range(6):
        step.out.zero_()
        step.conf.zero_()
        step.run(attn, vi["logits"], vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
        seen.append((step.out.clone(), step.conf.clone()))
    for out, conf in seen:
        assert torch.equal(out, seen[0][0]) and torch.equal(conf, seen[0][1]) and bool((conf > 0).all())
        assert bool((out.float().abs().amax(-1) > 0).all())


@pytest.mark.parametrize("kw,rows", [(dict(B=8, Nc=300, Hq=4, Hkv=2, V=32000), 160), (dict(B=8, Nc=300, Hq=4, Hkv=2, V=32000), 0),
                                     (dict(dtype="f32", d=64, B=16, Hq=4, Hkv=4, Nc=100, V=4096), 0)])
def test_step_with_logits_for_fewer_rows_than_the_tree_has(kw, rows):
    # a padded tree's unused nodes need no logits: their rows of the outputs stay; without any logits there is no vocabulary pass
    # and the attention must not start before what the caller enqueued in front of the step (here: its queries)
    cfg = W.small(W.CONFIGS["cfg2"], name="case", **kw)
    attn, vi = W.attention_inputs(cfg, DEV), W.verify_inputs(cfg, DEV)
    one, three = VerifyStep.for_config(cfg, DEV), VerifyStep.for_config(cfg, DEV)
    q = attn["q"].clone()
    for st in (one, three):
        st.conf.fill_(0.25)
        st.topk_idx.fill_(3)
    for i in range(4):
        torch.cuda._sleep(200000)
        attn["q"].copy_(q if i % 2 else -q)
        a = one.run(attn, vi["logits"][:rows], vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
        out = one.out.clone()
        three.attention(attn["q"], attn["k_cache"], attn["v_cache"], attn["k_draft"], attn["v_draft"], attn["sm_scale"])
        three.confidence_topk(vi["logits"][:rows])
        b = three.accept(vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
        assert torch.equal(out, three.out) and torch.equal(one.conf, three.conf) and torch.equal(one.topk_idx, three.topk_idx)
        assert bool((one.conf[rows:] == 0.25).all()) and all(torch.equal(a[key], b[key]) for key in a)


FIRST_CALL = """
import hashlib, sys
import torch
from paper_2608_27514_b200 import workloads as W
from paper_2608_27514_b200.step import VerifyStep
first, d = sys.argv[1], int(sys.argv[2])
cfg = W.small(W.CONFIGS["cfg2"], name="case", B=4, Nc=5056, Hq=28, Hkv=4, V=4096, d=d)
attn, vi = W.attention_inputs(cfg, "cuda:0"), W.verify_inputs(cfg, "cuda:0")
step = VerifyStep.for_config(cfg, "cuda:0")
if first == "step":
    step.run(attn, vi["logits"], vi["parent"], vi["state"], vi["mask_id"], cfg.tau)
    torch.cuda.synchronize()
    step.out.zero_()
step.attention(*(attn[k] for k in ("q", "k_cache", "v_cache", "k_draft", "v_draft", "sm_scale")))
print(hashlib.sha1(step.out.view(torch.int16).cpu().numpy().tobytes()).hexdigest())
"""


@pytest.mark.parametrize("d", [64, 128])
def test_results_do_not_depend_on_the_entry_point_that_ran_first(d):
    # whether items are cut over clusters is asked of the runtime once per process: the answer, and with it the order of the sums,
    # has to be the same whichever call asks first (a fresh process each)
    seen = {subprocess.run([sys.executable, "-c", FIRST_CALL, first, str(d)], check=True, capture_output=True, text=True, timeout=300).stdout
            for first in ("step", "attention")}
    assert len(seen) == 1
