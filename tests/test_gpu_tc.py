"""Parity of the tensor-core path (tcgen05 GEMMs; shapes with head_dim 128) against the oracle,
on sizes that span several weight tiles, k-blocks, column blocks and ragged tails."""
import numpy as np
import pytest
import torch

from oracle import adapters
from oracle import depcap_oracle as O
from paper_2604_15750_b200 import inputs
from paper_2604_15750_b200.binding import DC_ERR_NUMERIC

from parity import Case, compare

pytestmark = pytest.mark.gpu


def _wl(batch, n_q=4, n_kv=2, d=256, ff=512, vocab=2048, layers=2, ctx=(40, 128), last=16, win=32):
    return inputs.Workload(f"tc_b{batch}", layers, d, n_q, n_kv, 128, ff, vocab, "bf16", batch,
                           ctx[0], ctx[1], last, win, 64, 9000 + batch)


@pytest.mark.parametrize("batch", [1, 2, 3, 6])
def test_tc_small_models_match_the_oracle(batch):
    """M = 2 * batch * 48 activation rows: 96, 192, 288 (two column blocks), 576 (three)."""
    case = Case(_wl(batch), steer=None)
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    near, worst = compare(case, gpu, ora)
    eng.close()


def test_tc_ragged_lengths_and_steering():
    wl = _wl(3)
    lengths = dict(ctx_len=[128, 40, 77], last_len=[16, 5, 0], win_len=[32, 17, 9],
                   remain_len=[64, 17, 30])
    case = Case(wl, lengths=lengths, n_decoded=3, steer="decay")
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()


def test_tc_wider_model_many_tiles():
    """d_model 1024 (16 k-blocks, split-K on the O and down projections), d_ff 2816 (22 tiles)."""
    wl = _wl(2, n_q=8, n_kv=8, d=1024, ff=2816, vocab=4096, layers=3)
    case = Case(wl)
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()


def test_tc_and_cuda_core_paths_agree():
    """Same inputs through both kernel families (a debugging aid, not the parity claim)."""
    case = Case(_wl(2), steer="decay")
    e1, e2 = case.make_engine(impl=0), case.make_engine(impl=1)
    a, b = case.run_gpu(e1), case.run_gpu(e2)
    W = 32
    assert np.abs(a["lse"][:2, :W] - b["lse"][:2, :W]).max() < 2e-2
    assert np.array_equal(a["pred_id"][:2, :W], b["pred_id"][:2, :W])
    e1.close(); e2.close()


def test_tc_cache_beyond_ctx_len_may_hold_nan():
    wl = _wl(3)
    lengths = dict(ctx_len=[128, 41, 7], last_len=[16, 16, 3], win_len=[32, 30, 32],
                   remain_len=[64, 64, 64])
    case = Case(wl, lengths=lengths)
    eng = case.make_engine(max_batch=4, max_ctx=192)
    gpu, ora = case.run_gpu(eng, poison=True), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()


def test_tc_more_than_128_active_rows_and_long_context():
    """R = 32 + 128 = 160 active rows: two query tiles and two active key tiles; 5 context tiles."""
    wl = _wl(2, ctx=(513, 600), last=32, win=128)
    case = Case(wl)
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng, poison=True), case.run_oracle()
    compare(case, gpu, ora)
    eng.close()


def test_tc_attention_scores_far_above_those_of_the_first_key_tile():
    """The attention kernel fixes a row's reference point from its first key tile and runs a second
    pass when a later score lies more than 2^100 above it.  Three cached keys behind the first tile
    are scaled by 2000: for the rows whose query points their way they dominate by hundreds of log2
    units (one of them takes all the weight), for the others they vanish; with R = 160 active rows
    both the one-variant tiles and the packed tile of both variants go through it."""
    wl = _wl(2, ctx=(300, 300), last=32, win=128)
    case = Case(wl)
    for pos in (150, 210, 290):
        case.k_log[:, :, :, pos, :] *= 2000.0
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    eng.close()
    # Scores of several hundred log2 units turn a last-place difference in a rotated query into a
    # visible shift of weight between two keys, so the difference of the two variants (I_k) is
    # compared at 2e-2 absolute here instead of the 1e-3 of the well-conditioned cases; the
    # per-variant quantities keep their usual tolerance.
    for b in range(2):
        W = case.len["win_len"][b]
        for name in ("conf", "entropy", "lse"):
            ref = ora[b][name]
            err = np.abs(gpu[name][b, :W] - ref) / np.maximum(np.abs(ref), 1.0)
            assert np.isfinite(gpu[name][b, :W]).all() and err.max() <= 2e-2, (name, b, err.max())
        assert np.abs(gpu["influence"][b, :W] - ora[b]["influence"]).max() <= 2e-2
        assert (gpu["pred_id"][b, :W] == ora[b]["pred"]).mean() >= 0.95


def test_fused_dense_chain_is_the_path_taken_when_the_rows_fit_one_block():
    """M = 2 * 2 * 48 = 192 activation rows: the persistent dense chain must run (one launch that
    starts the step plus one per layer), not the per-op kernels; with 3 * 48 * 2 = 288 rows the
    per-op kernels run."""
    for batch, fused in ((2, True), (3, False)):
        case = Case(_wl(batch))
        eng = case.make_engine()
        di = case.device_inputs(eng)
        _, launches = eng.step_profiled(**di)
        if fused:
            assert launches["dense"] == case.n_layers + 1 and launches["qkv"] == 0
        else:
            assert launches["dense"] == 0 and launches["qkv"] == case.n_layers
        eng.close()


@pytest.mark.parametrize("n_q,n_kv,d,ff,last,win,influence", [
    (3, 1, 384, 640, [16] * 3, [32] * 3, True),                          # odd tile counts: no CTA pairs; 288 rows
    (40, 20, 512, 1024, [16] * 5 + [5], [32, 30, 20, 18, 27, 27], False),  # 272 rows: a last column block with fewer
    (40, 20, 512, 7680, [16] * 3, [128, 100, 47], True),                 # 672 rows, more units than CTA pairs
    (2, 2, 2176, 256, [16] * 3, [32] * 3, True),                         # norms of wide rows, with K splits folded in
    (2, 2, 4224, 256, [16] * 3, [32] * 3, True),
])
def test_tc_gemms_one_launch_each(n_q, n_kv, d, ff, last, win, influence):
    """Above 256 rows every GEMM is a launch of its own: column blocks of other widths, single CTAs and pairs,
    and units that take an accumulator after another one, at the tolerances of the other paths."""
    B = len(last)
    wl = _wl(B, n_q=n_q, n_kv=n_kv, d=d, ff=ff, last=max(last), win=max(win))
    case = Case(wl, lengths=dict(ctx_len=[40] * B, last_len=last, win_len=win, remain_len=[128] * B))
    eng = case.make_engine(max_window=(max(win) + 15) // 16 * 16)
    gpu, ora = case.run_gpu(eng, influence=influence), case.run_oracle(influence=influence)
    compare(case, gpu, ora)
    _, launches = eng.step_profiled(influence=influence, **case.device_inputs(eng))
    assert launches["dense"] == 0 and launches["qkv"] == case.n_layers
    eng.close()


@pytest.mark.parametrize("last,win,influence,rows", [(32, 96, True, 256), (0, 16, True, 32), (0, 32, False, 32),
                                                     (0, 7, False, 16), (0, 16, False, 16), (0, 40, False, 48)])
def test_fused_chain_at_its_row_limits(last, win, influence, rows):
    """The fused chain takes 16 .. 256 activation rows: both ends, against the oracle."""
    wl = _wl(1, last=max(last, 1), win=win)
    lengths = dict(ctx_len=[100], last_len=[last], win_len=[win], remain_len=[128])
    case = Case(wl, lengths=lengths)
    eng = case.make_engine(max_window=(win + 15) // 16 * 16)
    di = case.device_inputs(eng)
    out = eng.step(influence=influence, boundary=True, **di)
    sel = eng.select(di["win_ids"], di["win_len"])
    eng.synchronize()
    gpu = {k_: v_.cpu().numpy() for k_, v_ in out.items()}
    gpu.update({k_: v_.cpu().numpy() for k_, v_ in sel.items()})
    compare(case, gpu, case.run_oracle(influence=influence))
    _, launches = eng.step_profiled(influence=influence, boundary=True, **di)
    assert launches["dense"] == case.n_layers + 1, rows
    eng.close()


@pytest.mark.parametrize("n_q,n_kv,d", [(40, 20, 512), (28, 4, 512), (6, 2, 512), (40, 20, 2560), (28, 4, 1280)])
def test_fused_chain_qkv_helper_layouts(n_q, n_kv, d):
    """The QKV phase with 80, 36 (Dream's head counts) and 10 tiles.  Helper CTA pairs hand their sums over in the
    workspace of the K splits, which has room for that from d = 32 * tiles on: at d 512 only the 10 tiles have helpers; at
    d 2560 80 tiles have 34 helper pairs, six of which serve two tile pairs, at d 1280 36 have one each and some left over."""
    wl = _wl(1, n_q=n_q, n_kv=n_kv, d=d, ff=1024, vocab=2048, layers=2)
    case = Case(wl)
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng), case.run_oracle()
    compare(case, gpu, ora)
    di = case.device_inputs(eng)
    _, launches = eng.step_profiled(**di)
    assert launches["dense"] == case.n_layers + 1
    eng.close()


@pytest.mark.parametrize("ff,last,win,influence", [(7040, 32, 96, True), (7040, 0, 16, False), (4864, 16, 32, True)])
def test_fused_chain_gate_up_tile_heights(ff, last, win, influence):
    """Gate / up tiles of fewer than 128 rows: d_ff 7040 in 147 tiles of 48 (the 148th lies beyond the
    matrix), 4864 in 122 of 40 with a remainder; 256, 16 and 96 activation rows."""
    wl = _wl(1, ff=ff, last=max(last, 1), win=win)
    lengths = dict(ctx_len=[100], last_len=[last], win_len=[win], remain_len=[128])
    case = Case(wl, lengths=lengths)
    eng = case.make_engine(max_window=win)
    di = case.device_inputs(eng)
    out = eng.step(influence=influence, boundary=True, **di)
    sel = eng.select(di["win_ids"], di["win_len"])
    eng.synchronize()
    gpu = {k_: v_.cpu().numpy() for k_, v_ in out.items()}
    gpu.update({k_: v_.cpu().numpy() for k_, v_ in sel.items()})
    compare(case, gpu, case.run_oracle(influence=influence))
    _, launches = eng.step_profiled(influence=influence, boundary=True, **di)
    assert launches["dense"] == case.n_layers + 1
    eng.close()


@pytest.mark.parametrize("n_q,n_kv,ctx,last,win", [
    (4, 2, [0], [0], [16]),                  # active keys only
    (4, 2, [1], [1], [1]),                   # one cached key; two rows
    (4, 2, [128], [0], [7]),                 # whole context tile
    (4, 4, [129], [5], [27]),                # one key in the second tile, 32 rows, append at an odd position
    (4, 2, [700], [31], [33]),               # 64 rows: two row tiles; six tiles through the deep ring
    (4, 2, [40, 64, 7], [16, 0, 5], [32, 3, 12]),   # 48, 16 and 32 rows, one sequence behind the other
    (40, 20, [513, 40, 300, 250], [16, 5, 0, 9], [32, 17, 9, 24]),   # more CTAs than SMs: two on an SM
    (32, 32, [1200, 1163, 1126, 1000, 960, 1190, 900, 1024], [0] * 8, [24, 19, 14, 9, 32, 8, 24, 1]),   # as above, caches larger than L2
])
def test_tc_attention_few_rows(n_q, n_kv, ctx, last, win):
    """One variant of few rows: keys on the lanes, 32 rows a CTA.  With the last block
    appended: its keys and values at the 2e-2 of a bf16 stack, nothing else of the cache written."""
    B = len(ctx)
    wl = _wl(B, n_q=n_q, n_kv=n_kv, ctx=(max(max(ctx), 1), max(max(ctx), 1)), last=max(max(last), 1), win=max(win))
    case = Case(wl, lengths=dict(ctx_len=ctx, last_len=last, win_len=win, remain_len=[64] * B))
    eng = case.make_engine(max_ctx=1280, max_window=(max(win) + 15) // 16 * 16)
    di = case.device_inputs(eng, poison=True)
    k0, v0 = di["k_cache"].clone(), di["v_cache"].clone()
    out = eng.step(influence=False, boundary=True, export_kv=True, **di)
    sel = eng.select(di["win_ids"], di["win_len"])
    eng.synchronize()
    gpu = {k_: v_.cpu().numpy() for k_, v_ in {**out, **sel}.items()}
    ora = {b: O.step(case.ocfg, case.ow, adapters.to_np(case.k_log[:, b]), adapters.to_np(case.v_log[:, b]), ctx[b],
                     case.last_ids[b, :last[b]].numpy(), case.win_ids[b, :win[b]].numpy(), 64, influence=False,
                     return_kv=True) for b in range(B)}
    compare(case, gpu, ora)
    for b in range(B):
        end = ctx[b] + last[b]
        for new, old in ((di["k_cache"][:, b], k0[:, b]), (di["v_cache"][:, b].transpose(-1, -2), v0[:, b].transpose(-1, -2))):
            assert torch.equal(new[:, :, :ctx[b]], old[:, :, :ctx[b]]) and new[:, :, end:].isnan().all()
            which = 0 if new.data_ptr() == di["k_cache"][:, b].data_ptr() else 1
            for l in range(case.n_layers if last[b] else 0):
                ref = ora[b]["kv_last"][l][which]                    # [last, nkv, hd]
                got = new[l, :, ctx[b]:end].float().permute(1, 0, 2).cpu().numpy()
                assert np.abs(got - ref).max() / max(np.abs(ref).max(), 1.0) <= 2e-2, (b, l)
    eng.close()


@pytest.mark.parametrize("batch,ctx,last,win", [
    (2, [300, 300], [32, 32], [128, 128]),                 # two query tiles, the second of both variants
    (4, [128, 40, 77, 0], [16, 5, 0, 9], [32, 17, 9, 27]), # both variants in one tile, ragged
    (1, [513], [32], [96]),                                # 128 rows a variant
])
def test_tc_attention_many_heads(batch, ctx, last, win):
    """40 heads: more (row tile, head) units than the few-rows kernel is given, so rows on the lanes.  Poisoned
    caches, and cached keys (where there are 300) that make the pass run again."""
    wl = _wl(batch, n_q=40, n_kv=20, ctx=(max(ctx), max(ctx)), last=max(last), win=max(win))
    case = Case(wl, lengths=dict(ctx_len=ctx, last_len=last, win_len=win, remain_len=[128] * batch))
    eng = case.make_engine(max_window=(max(win) + 15) // 16 * 16)
    gpu, ora = case.run_gpu(eng, poison=True), case.run_oracle()
    compare(case, gpu, ora)
    if ctx[0] == 300:
        for pos in (150, 210, 290):
            case.k_log[:, :, :, pos, :] *= 2000.0
        gpu, ora = case.run_gpu(eng), case.run_oracle()
        for b in range(batch):   # (tolerances as in the test above of scores far from the first)
            W = win[b]
            for name in ("conf", "entropy", "lse"):
                ref = ora[b][name]
                assert (np.abs(gpu[name][b, :W] - ref) / np.maximum(np.abs(ref), 1.0)).max() <= 2e-2, (name, b)
            assert (gpu["pred_id"][b, :W] == ora[b]["pred"]).mean() >= 0.95
    eng.close()


def test_tc_attention_few_rows_with_scores_far_above_the_first():
    """Keys behind the first 32 that lie hundreds of log2 units above them: the passes that find the maxima and
    use them.  Tolerances as in the test of the other kernel above."""
    wl = _wl(2, ctx=(300, 300), last=1, win=40)
    case = Case(wl, lengths=dict(ctx_len=[300, 290], last_len=[0, 0], win_len=[40, 33], remain_len=[64, 64]))
    for pos in (50, 150, 270):
        case.k_log[:, :, :, pos, :] *= 2000.0
    eng = case.make_engine()
    gpu, ora = case.run_gpu(eng, influence=False), case.run_oracle(influence=False)
    eng.close()
    for b in range(2):
        W = case.len["win_len"][b]
        for name in ("conf", "entropy", "lse"):
            ref = ora[b][name]
            err = np.abs(gpu[name][b, :W] - ref) / np.maximum(np.abs(ref), 1.0)
            assert np.isfinite(gpu[name][b, :W]).all() and err.max() <= 2e-2, (name, b, err.max())
        assert (gpu["pred_id"][b, :W] == ora[b]["pred"]).mean() >= 0.95


@pytest.mark.parametrize("n_q,n_kv,influence", [
    (4, 2, False), (4, 2, True),     # keys on the lanes, one variant and two
    (40, 20, True),                  # rows on the lanes, both variants in one tile
])
def test_tc_non_finite_keys_of_one_sequence_stay_there(n_q, n_kv, influence):
    """A sequence whose cached keys and values hold NaN inside ctx_len (and whose own rows become NaN with
    them): the sequences before and behind it in the batch give the bits of a clean run, and so does a smaller
    step afterwards, whose last key tile ends in (57 rows, padded to 64) and reads on into rows that the NaN step
    left in the workspace."""
    wl = _wl(3, n_q=n_q, n_kv=n_kv)
    case = Case(wl, lengths=dict(ctx_len=[40, 77, 128], last_len=[16, 16, 3], win_len=[21, 30, 17], remain_len=[64] * 3))
    eng, ref = case.make_engine(max_window=48), case.make_engine(max_window=48)

    def step(e, di, seqs, **other):
        args = {k_: v_[:seqs] if isinstance(v_, list) else v_ for k_, v_ in di.items()}
        out = e.step(influence=influence, boundary=True, **{**args, **other})
        e.synchronize()
        return {k_: v_.cpu().numpy() for k_, v_ in out.items()}

    di = case.device_inputs(eng)
    clean = step(ref, di, 3)
    bad = dict(di, k_cache=di["k_cache"].clone(), v_cache=di["v_cache"].clone())
    bad["k_cache"][:, 1, :, 5] = float("nan")
    bad["v_cache"][:, 1, :, :, 9] = float("nan")
    got = step(eng, bad, 3)
    assert got["status"][[0, 2]].tolist() == [0, 0] and got["status"][1] == DC_ERR_NUMERIC
    for b in (0, 2):
        W = case.len["win_len"][b]
        for k_ in ("pred_id", "conf", "entropy", "lse", "influence"):
            assert np.array_equal(got[k_][b, :W], clean[k_][b, :W]), (k_, b)
    small, again = (step(e, di, 1, win_len=[41]) for e in (ref, eng))
    for k_ in ("pred_id", "conf", "entropy", "lse", "influence"):
        assert np.array_equal(small[k_][0, :41], again[k_][0, :41]), k_
    assert again["status"][0] == 0
    eng.close(); ref.close()


@pytest.mark.parametrize("ff,win,influence", [(512, 16, False), (640, 32, True)])
def test_norm_gains_on_8_byte_boundaries(ff, win, influence):
    """The fused chain brings the gains in by bulk copies, which start on 16-byte boundaries; gains on 8-byte
    boundaries keep the launch per operation (16 rows; 64 rows with an odd number of gate / up tiles)."""
    wl = _wl(1, ff=ff, last=1, win=win)
    case = Case(wl, lengths=dict(ctx_len=[100], last_len=[0], win_len=[win], remain_len=[128]))
    for lw in case.weights["layers"]:
        for k_ in ("norm1", "norm2"):
            at = torch.zeros(wl.d_model + 4, dtype=torch.bfloat16, device="cuda:0")[4:]
            lw[k_] = at.copy_(lw[k_])
    eng = case.make_engine(max_window=win)
    assert eng._weights["layers"][0]["norm1"].data_ptr() % 16 == 8
    di = case.device_inputs(eng)
    out = eng.step(influence=influence, boundary=True, **di)
    sel = eng.select(di["win_ids"], di["win_len"])
    eng.synchronize()
    gpu = {k_: v_.cpu().numpy() for k_, v_ in {**out, **sel}.items()}
    compare(case, gpu, case.run_oracle(influence=influence))
    _, launches = eng.step_profiled(influence=influence, boundary=True, **di)
    assert launches["dense"] == 0 and launches["qkv"] == case.n_layers
    eng.close()


@pytest.mark.parametrize("d,xlogp", [(12288, True), (12416, False)])
def test_rows_that_do_not_fit_without_a_shared_memory_opt_in(d, xlogp):
    """Models wider than 48 KB of fp32 a row: the rows of the LM head, with and without the cross log-probs (which
    stage a row of 48 KB at most), and the rows that a later step carries."""
    wl = inputs.Workload("tc_wide", 1, d, 2, 2, 128, 256, 512, "bf16", 1, 40, 40, 3, 16, 32, 77)
    case = Case(wl)
    eng = case.make_engine()
    di = case.device_inputs(eng)
    h = torch.zeros((1, eng.max_window, d), dtype=torch.bfloat16, device=eng.device)
    out = eng.step(influence=True, boundary=True, want_xlogp=xlogp, h_out=h, **di)
    eng.synchronize()
    assert int(out["status"][0]) == 0
    ora = case.run_oracle()[0]
    for name in ("conf", "entropy", "lse"):
        got = out[name][0, :16].cpu().numpy()
        assert (np.abs(got - ora[name]) / np.maximum(np.abs(ora[name]), 1.0)).max() <= 2e-2, name
    if xlogp:
        got = out["xlogp"][0, :16, :16].cpu().numpy()
        same = out["pred_id"][0, :16].cpu().numpy() == ora["pred"]
        assert same.mean() >= 0.9
        err = np.abs(got - ora["xlogp"]) / np.maximum(np.abs(ora["xlogp"]), 1.0)
        assert err[:, same].max() <= 2e-2
    assert np.abs(h[0, :16].float().cpu().numpy()).max() > 0 and torch.isfinite(h).all()
    eng.close()
