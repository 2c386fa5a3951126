"""CUDA-core kernels at the shapes where their tiles can go wrong, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import adapters
from oracle import depcap_oracle as O
from paper_2604_15750_b200 import inputs
from paper_2604_15750_b200.binding import DC_ERR_NUMERIC

from parity import Case, compare

pytestmark = pytest.mark.gpu


def _fused(eng, case):
    """whether a step of the case runs as one launch"""
    _, launches = eng.step_profiled(**case.device_inputs(eng, poison=case.wl.ctx_max > 0))
    assert (launches["dense"] == 1) == (launches["qkv"] == 0) and launches["dense"] <= 1
    return launches["dense"] == 1


def _wl(name, dtype, n_q, n_kv, hd, d, ff, vocab, batch, ctx, last, win):
    return inputs.Workload(name, 2, d, n_q, n_kv, hd, ff, vocab, dtype, batch, ctx[0], ctx[1], last, win, 64, 31337)


@pytest.mark.parametrize("wl", [
    # every GEMM above the small-tile limit (64 x 64 tiles), M 768 not a multiple of what a tile holds in N
    _wl("simt_large", "f32", 4, 2, 64, 512, 1404, 3001, 3, (50, 90), 24, 96),
    # one row tile, K 1024 and more chunks than the ring has stages; fewer features than a tile
    _wl("simt_small", "f32", 3, 1, 96, 132, 1028, 130, 1, (0, 0), 3, 5),
    # head_dim not a multiple of 32: rotation outside the GEMM; rows that are not 16-byte aligned
    _wl("simt_odd", "bf16", 4, 2, 20, 36, 50, 1003, 2, (17, 40), 7, 19),
    # head_dim not a multiple of 4, attention tiles with a remainder in both segments
    _wl("simt_hd6", "f32", 2, 2, 6, 64, 72, 509, 2, (65, 129), 33, 40),
    # bf16 with tiles of both kinds and long contexts
    _wl("simt_bf16", "bf16", 4, 4, 32, 256, 520, 4100, 2, (200, 331), 16, 48),
    # heads whose tiles do not fit in shared memory: more than one tile of cached keys, and of active ones
    _wl("simt_hd4096", "f32", 2, 1, 4096, 64, 72, 130, 2, (5, 300), 40, 240),
    _wl("simt_hd6000", "bf16", 1, 1, 6000, 64, 72, 130, 1, (30, 30), 3, 17),
], ids=lambda w: w.name)
def test_cuda_core_shapes(wl):
    case = Case(wl, ctx_from_oracle=wl.dtype == "f32" and wl.ctx_max > 0, steer="decay")
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng, poison=wl.ctx_max > 0), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()
    raw = Case(wl, ctx_from_oracle=wl.dtype == "f32" and wl.ctx_max > 0)   # the stack's own rows at the LM head
    eng = raw.make_engine()
    gpu, ora = raw.run_gpu(eng, poison=wl.ctx_max > 0), raw.run_oracle()
    compare(raw, gpu, ora)
    eng.close()


@pytest.mark.parametrize("wl", [
    # head_dim 128 (tiles of 32 keys), d not a multiple of the k-chunk, one context tile with a remainder
    _wl("fused_hd128", "f32", 2, 1, 128, 260, 388, 515, 2, (33, 70), 5, 21),
    # bf16, head_dim 96, the widest row a warp norms that still fits, two rounds of tiles
    _wl("fused_bf16", "bf16", 4, 2, 96, 1024, 520, 2048, 2, (1, 65), 16, 40),
    # three sequences, no context for one, MLP of several k-chunks
    _wl("fused_ragged", "f32", 4, 4, 32, 128, 1160, 1031, 3, (0, 130), 9, 48),
], ids=lambda w: w.name)
def test_fused_step_and_separate_launches(wl):
    """The one-launch step against the oracle, and the same step as separate launches (fp32 sums in
    another order: 1e-5 relative to the largest value; bf16 rounds between the stages: 2e-2)."""
    lengths = dict(ctx_len=[wl.ctx_max, 0, wl.ctx_min][:wl.batch], last_len=[wl.last_len, 3, 0][:wl.batch],
                   win_len=[wl.win_len, 1, 17][:wl.batch], remain_len=[64, 8, 30][:wl.batch])
    case = Case(wl, lengths=lengths, n_decoded=0)
    eng = case.make_engine()
    assert _fused(eng, case)
    gpu, ora = case.run_gpu(eng, poison=True), case.run_oracle()
    compare(case, gpu, ora)
    eng.step_profiled(**case.device_inputs(eng, poison=True))   # (the call that is profiled is the same one)
    for k in ("conf", "entropy", "lse", "influence", "block_len"):
        assert np.array_equal(eng.out[k].cpu().numpy(), gpu[k]), k
    eng.set_option(1, 0)                       # DC_OPT_COOPERATIVE off: one launch per operation
    assert not _fused(eng, case)
    one = case.run_gpu(eng, poison=True)
    tol = 1e-5 if wl.dtype == "f32" else 2e-2
    for b in range(wl.batch):
        n = lengths["win_len"][b]
        for k in ("conf", "entropy", "lse"):
            assert abs(gpu[k][b, :n] - one[k][b, :n]).max() <= tol * max(1.0, abs(one[k][b, :n]).max()), (k, b)
    eng.close()


@pytest.mark.parametrize("hd,cooperative,fused", [(32, 1, True), (32, 0, False), (16, 1, False)])
def test_ragged_rows_lie_behind_one_another(hd, cooperative, fused):
    """Sequences of 48, 16 and 32 rows (rounded up) in a batch, fp32: signals at 1e-4, the appended keys and values at
    1e-4, nothing else of the cache written.  The fused step, separate launches, and separate launches with the
    rotation outside the GEMM."""
    ctx, last, win = [40, 64, 7], [16, 0, 5], [32, 3, 12]
    wl = inputs.Workload("ragged_f32", 2, 64, 4, 2, hd, 128, 300, "f32", 3, 64, 64, 16, 32, 64, 515)
    case = Case(wl, lengths=dict(ctx_len=ctx, last_len=last, win_len=win, remain_len=[64] * 3))
    eng = case.make_engine(max_ctx=128)
    eng.set_option(1, cooperative)             # DC_OPT_COOPERATIVE
    assert _fused(eng, case) == fused
    di = case.device_inputs(eng)
    k0, v0 = di["k_cache"].clone(), di["v_cache"].clone()
    out = eng.step(influence=True, boundary=True, export_kv=True, **di)
    sel = eng.select(di["win_ids"], di["win_len"])
    eng.synchronize()
    gpu = {k_: v_.cpu().numpy() for k_, v_ in {**out, **sel}.items()}
    ora = {b: O.step(case.ocfg, case.ow, adapters.to_np(case.k_log[:, b]), adapters.to_np(case.v_log[:, b]), ctx[b],
                     case.last_ids[b, :last[b]].numpy(), case.win_ids[b, :win[b]].numpy(), 64, return_kv=True)
           for b in range(3)}
    compare(case, gpu, ora)
    for b in range(3):
        end = ctx[b] + last[b]
        for which, (new, old) in enumerate(((di["k_cache"][:, b], k0[:, b]),
                                            (di["v_cache"][:, b].transpose(-1, -2), v0[:, b].transpose(-1, -2)))):
            assert torch.equal(new[:, :, :ctx[b]], old[:, :, :ctx[b]]) and torch.equal(new[:, :, end:], old[:, :, end:])
            for l in range(2 if last[b] else 0):
                ref = ora[b]["kv_last"][l][which]                    # [last, nkv, hd]
                got = new[l, :, ctx[b]:end].permute(1, 0, 2).cpu().numpy()
                assert np.abs(got - ref).max() / max(np.abs(ref).max(), 1.0) <= 1e-4, (b, l)
    eng.close()


@pytest.mark.parametrize("cooperative", [1, 0])   # the fused step, separate launches
def test_position_whose_logits_are_all_minus_infinity(cooperative):
    """Not a confident position: confidence, entropy and log-sum-exp are NaN, so that no threshold is met, and the
    status says so; the other positions have the bits of a run without it."""
    wl = _wl("simt_minf", "f32", 4, 4, 32, 128, 256, 515, 1, (40, 40), 5, 16)
    case = Case(wl, steer="decay")
    case.weights["lm_head"][:, 0] = -1.0
    eng = case.make_engine()
    eng.set_option(1, cooperative)             # DC_OPT_COOPERATIVE
    di = case.device_inputs(eng)
    di["h_final"][..., 0] = 0.0

    def run():
        out = eng.step(influence=True, boundary=True, **di)
        sel = eng.select(di["win_ids"], [16], block_len=torch.full((1,), 16, dtype=torch.int32, device=eng.device))
        eng.synchronize()
        return {k_: v_.cpu().numpy()[0] for k_, v_ in {**out, **sel}.items()}

    clean = run()
    di["h_final"][0, :, 3] = 0.0
    di["h_final"][0, :, 3, 0] = float("inf")
    got = run()
    assert clean["status"] == 0 and got["status"] == DC_ERR_NUMERIC
    assert np.isnan([got[k_][3] for k_ in ("conf", "entropy", "lse")]).all()
    assert got["pred_id"][3] == wl.mask_id and got["influence"][3] == 0 and got["sel_mask"][3] == 0
    rest = np.arange(16) != 3
    for k_ in ("pred_id", "conf", "entropy", "lse", "influence"):
        assert np.array_equal(got[k_][rest], clean[k_][rest]), k_
    eng.close()


@pytest.mark.parametrize("d", [1028, 2052, 4100, 8196])
def test_norm_of_wide_rows(d):
    """RMSNorm as a launch of its own: a row in 2, 4 or 8 pieces of registers, with a remainder in the last, and
    wider ones."""
    wl = inputs.Workload(f"norm{d}", 1, d, 2, 2, 32, 64, 512, "f32", 1, 16, 16, 4, 16, 32, 900 + d % 7)
    case = Case(wl, steer=None)
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()
