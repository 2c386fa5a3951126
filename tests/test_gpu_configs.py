"""Parity at the row counts, batch sizes, context lengths and vocabulary of the larger benchmark
configurations (LLaDA-8B shape at batch 8 with ragged prompts, Dream-7B shape at batch 4, the
long-context LLaDA shape at batch 16), in the launch configuration bench.py times: the per-op
tensor-core kernels with the K splits the host picks for these shapes, 32 context tiles per
sequence at the long context, the LM head over 2048 / 512 / 4096 rows.

One transformer layer (the oracle cannot run more at these widths in seconds); every other
dimension is the workload's.  Sequences are independent, so the oracle runs sequences 0 and B-1.
Each configuration is compared twice: raw (the stack's own output feeds the LM head: every float
through the real shapes, decisions degenerate on random-init weights) and steered (shaped LM-head
inputs: ids, boundaries and subsets exercised at the full vocabulary).  The LM-head stage is also
held to I_k within 1e-3 absolute (plus under 1e-4 for the tensor core's accumulator) on rows the
GPU stack produced.
"""
import numpy as np
import pytest
import torch

from paper_2604_15750_b200 import inputs

from parity import Case, compare, lm_stage_strict

pytestmark = pytest.mark.gpu


def _run(name, profile, path, n_ctx_tiles):
    wl = inputs.scaled(inputs.WORKLOADS[name], n_layers=1)
    case = Case(wl, steer=profile)
    seqs = [0, wl.batch - 1]
    eng = case.make_engine()
    _, launches = eng.step_profiled(**case.device_inputs(eng))
    if path == "per-op":
        assert launches["dense"] == 0 and launches["qkv"] == 1 and launches["attn"] == 1
    assert launches["lmhead"] == 2                       # tensor-core LM head + combine
    assert max(case.len["ctx_len"]) > 128 * (n_ctx_tiles - 1)
    npos = sum(case.len["win_len"][b] for b in seqs)
    # steered: the decisions at the full vocabulary
    near, worst = compare(case, case.run_gpu(eng), case.run_oracle(seqs=seqs),
                          label=f"{name} x 1 layer, steered {profile}")
    assert near["pred"] <= npos // 10 and near["subset"] <= len(seqs) and near["block_len"] <= len(seqs)
    o0 = case.run_oracle(seqs=[0])[0]
    assert (o0["conf"] > 0.9).any()                      # the steering did shape the distributions
    # raw: the stack's own rows through the LM head
    steer, case.steer = case.steer, None
    near_r, worst_r = compare(case, case.run_gpu(eng), case.run_oracle(seqs=seqs),
                              label=f"{name} x 1 layer, raw")
    # the LM-head stage on those rows at the strict influence tolerance
    strict = lm_stage_strict(case, eng, seqs=seqs)
    assert strict["influence"] <= 1e-3
    case.steer = steer
    eng.close()
    return near, worst, near_r, worst_r, strict


def test_llada8b_batch8_ragged_prompts_full_rows():
    """B = 8, prompts of 768..1024 tokens (8 context tiles), R = 160 rows per variant: M = 2560
    activation rows (ten column blocks, split-K by the round model), 2048 LM-head rows."""
    _run("llada8b_b8", "decay", "per-op", 7)


def test_dream7b_batch4_grouped_heads_full_rows():
    """B = 4, 28 query / 4 KV heads, prompts of 768 tokens, M = 768 rows, V = 152064."""
    _run("dream7b_b4", "decay", "per-op", 6)


def test_llada8b_long_context_batch16_bimodal():
    """B = 16, 4096 cached keys per sequence (32 context tiles), M = 5120 rows, 4096 LM-head rows,
    max-probability bimodal (half the positions peaked above 0.9, half flat)."""
    near, worst, near_r, worst_r, strict = _run("llada8b_long", "bimodal", "per-op", 32)


@pytest.mark.parametrize("dtype,hd,win", [("f32", 32, 32), ("bf16", 128, 16), ("bf16", 128, 32)])
def test_a_stream_with_fewer_sms_than_the_device(dtype, hd, win):
    """The fused CUDA-core step and the dense chain need a CTA on every SM at once.  On a stream of 16 SMs their
    launches are refused, and the steps run as separate launches."""
    gc = pytest.importorskip("torch.cuda.green_contexts")
    if not gc.SUPPORTED:
        pytest.skip("no green contexts")
    wl = inputs.Workload("few_sms", 2, 256, 4, 2, hd, 512, 2048, dtype, 1, 100, 100, 16, win, 64, 31337)
    case = Case(wl)
    green = gc.GreenContext.create(16, 0)
    green.set_context()
    try:
        with torch.cuda.stream(green.Stream()):
            eng = case.make_engine()
            gpu = case.run_gpu(eng)
            _, launches = eng.step_profiled(**case.device_inputs(eng))
            eng.close()
    finally:
        green.pop_context()
    assert launches["dense"] == 0 and launches["qkv"] == case.n_layers
    compare(case, gpu, case.run_oracle())
