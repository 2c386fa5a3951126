"""Decision kernels fed exactly the floats the oracle gets: results must be bit-identical."""
import numpy as np
import pytest
import torch

from oracle import depcap_oracle as O
from paper_2604_15750_b200 import Hyper, inputs

from parity import Case

pytestmark = pytest.mark.gpu

WL = inputs.scaled(inputs.WORKLOADS["tiny_f32"], n_layers=0, batch=1)


def _engine(hyper, max_batch=32, max_window=128):
    case = Case(inputs.scaled(WL, ctx_min=0, ctx_max=0), n_layers=0, hyper=hyper)
    return case.make_engine(max_batch=max_batch, max_window=max_window, max_ctx=0)


def _ocfg(hp):
    return O.OracleConfig(n_layers=0, d_model=1, n_q_heads=1, n_kv_heads=1, head_dim=1, d_ff=1,
                          vocab=2, mask_id=1, lam=hp.lam, L_min=hp.L_min, L_max=hp.L_max,
                          smooth_radius=hp.smooth_radius, norm_mode=hp.norm_mode,
                          boundary_mode=hp.boundary_mode, cap_mode=hp.cap_mode)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("norm", [0, 1, 2])
@pytest.mark.parametrize("radius", [0, 1, 3])
def test_boundary_bit_exact(mode, norm, radius):
    hp = Hyper(boundary_mode=mode, norm_mode=norm, smooth_radius=radius, lam=1.2)
    eng = _engine(hp)
    r = np.random.default_rng(100 + 10 * mode + 3 * norm + radius)
    W, B = 128, 32
    for rep in range(8):
        win = r.integers(1, W + 1, B)
        remain = r.integers(1, 300, B)
        have = (r.random(B) < 0.9).astype(np.int32)
        I = (np.abs(r.standard_normal((B, W))) * np.exp(-np.arange(W) / r.uniform(2, 40))
             ).astype(np.float32)
        H = (r.random((B, W)) * r.uniform(0.1, 11)).astype(np.float32)
        if rep == 0:                       # adversarial: exact zeros, ties, tiny values
            I[:4] = 0.0
            H[4:8] = H[4:8, :1]
            I[8:12] *= 1e-30
            I[12:16] = H[12:16] * np.float32(1.2)
        out = eng.boundary(torch.from_numpy(I).cuda(), torch.from_numpy(H).cuda(), list(win),
                           list(remain), list(have))
        eng.synchronize()
        g = {k: v.cpu().numpy() for k, v in out.items()}
        for b in range(B):
            L, score, ci, cs = O.boundary(I[b], H[b], int(win[b]), int(remain[b]), bool(have[b]),
                                          _ocfg(hp))
            n = len(score)
            assert int(g["block_len"][b]) == L, (rep, b)
            assert np.array_equal(g["score"][b, :n].view(np.uint32), score.view(np.uint32))
            assert np.array_equal(g["cum_influence"][b, :n].view(np.uint32), ci.view(np.uint32))
            assert np.array_equal(g["cum_score"][b, :n].view(np.uint32), cs.view(np.uint32))
    eng.close()


@pytest.mark.parametrize("cap_mode", [0, 1])
def test_select_bit_exact(cap_mode):
    hp = Hyper(cap_mode=cap_mode)
    eng = _engine(hp)
    r = np.random.default_rng(7 + cap_mode)
    W, B = 128, 32
    mask_id = WL.mask_id
    total = 0
    for rep in range(12):
        win = r.integers(1, W + 1, B)
        blk = np.array([r.integers(0, w + 1) for w in win]).astype(np.int32)
        conf = r.random((B, W)).astype(np.float32)
        if rep % 3 == 0:
            conf = (0.6 + 0.4 * r.random((B, W))).astype(np.float32)          # big pools
        if rep % 4 == 1:
            conf = np.round(conf, 1).astype(np.float32)                        # many ties
            conf[:, ::7] = np.float32(0.8); conf[:, ::11] = np.float32(0.95)   # on thresholds
        x = (r.standard_normal((B, W, W)) * 6 - 9).astype(np.float32)
        if rep % 4 == 2:
            x[:, :, :] = np.float32(-8.0)                                      # D == gamma exactly
        ids = np.where(r.random((B, W)) < 0.8, mask_id, 5).astype(np.int32)
        out = eng.select(torch.from_numpy(ids).cuda(), list(win),
                         conf=torch.from_numpy(conf).cuda(), xlogp=torch.from_numpy(x).cuda(),
                         block_len=torch.from_numpy(blk).cuda())
        eng.synchronize()
        g = {k: v.cpu().numpy() for k, v in out.items()}
        for b in range(B):
            w = int(win[b])
            want = O.cap_select(conf[b, :w], ids[b, :w] == mask_id, x[b, :w, :w], int(blk[b]),
                                hp.tau_low, hp.tau_high, hp.gamma, cap_mode)
            n = int(g["sel_count"][b])
            assert list(g["sel_idx"][b, :n]) == want, (rep, b)
            assert [i for i in range(w) if g["sel_mask"][b, i]] == want
            total += n
    assert total > 500
    eng.close()


def test_select_threshold_override_reduces_to_the_baselines():
    eng = _engine(Hyper())
    r = np.random.default_rng(3)
    W, B = 64, 4
    conf = r.random((B, 128)).astype(np.float32)
    x = (r.standard_normal((B, 128, 128)) * 6 - 9).astype(np.float32)
    ids = np.full((B, 128), WL.mask_id, dtype=np.int32)
    blk = np.full(B, W, dtype=np.int32)
    args = dict(conf=torch.from_numpy(conf).cuda(), xlogp=torch.from_numpy(x).cuda(),
                block_len=torch.from_numpy(blk).cuda())
    # tau_low above 1: one token per step, the most confident one
    g = eng.select(torch.from_numpy(ids).cuda(), [W] * B, thresholds=(1.5, 2.0, -16.0), **args)
    eng.synchronize()
    assert list(g["sel_count"].cpu().numpy()[:B]) == [1] * B
    assert list(g["sel_idx"][:B, 0].cpu().numpy()) == list(conf[:, :W].argmax(axis=1))
    # gamma = +inf: plain confidence thresholding at 0.9
    g = eng.select(torch.from_numpy(ids).cuda(), [W] * B, thresholds=(0.9, 0.95, float("inf")),
                   **args)
    eng.synchronize()
    m = g["sel_mask"].cpu().numpy()[:B, :W]
    assert np.array_equal(m.astype(bool), conf[:, :W] >= np.float32(0.9))
    eng.close()


def test_batched_decisions_8192_sequences_bit_exact_on_a_sample():
    """dc_boundary_batched / dc_select_batched over 8192 sequences with device-side length
    arrays (the shape bench.py --mode decisions times): 96 sampled sequences, bit for bit."""
    hp = Hyper()
    eng = _engine(hp, max_batch=1, max_window=128)
    r = np.random.default_rng(2024)
    W, B = 128, 8192
    mask_id = WL.mask_id
    win = r.integers(1, W + 1, B).astype(np.int32)
    remain = r.integers(1, 300, B).astype(np.int32)
    have = (r.random(B) < 0.9).astype(np.int32)
    I = (np.abs(r.standard_normal((B, W))) * np.exp(-np.arange(W) / 16.0)).astype(np.float32)
    H = (r.random((B, W)) * 8).astype(np.float32)
    conf = np.where(r.random((B, W)) < 0.5, 0.9 + 0.1 * r.random((B, W)), r.random((B, W))).astype(np.float32)
    x = (r.standard_normal((B, W, W)) * 6 - 12).astype(np.float32)
    ids = np.where(r.random((B, W)) < 0.8, mask_id, 5).astype(np.int32)
    dev = eng.device
    t = lambda a: torch.from_numpy(a).to(dev)
    bo = dict(score=torch.zeros((B, W), device=dev), cum_influence=torch.zeros((B, W), device=dev),
              cum_score=torch.zeros((B, W), device=dev),
              block_len=torch.zeros((B,), dtype=torch.int32, device=dev))
    eng.boundary_batched(t(I), t(H), t(win), t(remain), bo, have_prev=t(have))
    so = dict(sel_mask=torch.zeros((B, W), dtype=torch.uint8, device=dev),
              sel_idx=torch.zeros((B, W), dtype=torch.int32, device=dev),
              sel_count=torch.zeros((B,), dtype=torch.int32, device=dev))
    eng.select_batched(t(conf), t(ids), t(x), bo["block_len"], t(win), so)
    eng.synchronize()
    g = {k: v.cpu().numpy() for k, v in {**bo, **so}.items()}
    picked = 0
    for b in list(range(32)) + list(r.integers(0, B, 62)) + [B - 2, B - 1]:
        L, score, ci, cs = O.boundary(I[b], H[b], int(win[b]), int(remain[b]), bool(have[b]), _ocfg(hp))
        n = len(score)
        assert int(g["block_len"][b]) == L, b
        assert np.array_equal(g["score"][b, :n].view(np.uint32), score.view(np.uint32))
        assert np.array_equal(g["cum_score"][b, :n].view(np.uint32), cs.view(np.uint32))
        w = int(win[b])
        want = O.cap_select(conf[b, :w], ids[b, :w] == mask_id, x[b, :w, :w], L, hp.tau_low,
                            hp.tau_high, hp.gamma, hp.cap_mode)
        cnt = int(g["sel_count"][b])
        assert list(g["sel_idx"][b, :cnt]) == want, b
        picked += cnt
    assert picked > 96
    eng.close()


@pytest.mark.parametrize("W,B,cap_mode", [(16, 3, 1), (64, 700, 0), (80, 593, 1), (256, 601, 0), (256, 2, 1)])
def test_decisions_one_warp_per_sequence_bit_exact(W, B, cap_mode):
    """Two, four and eight positions per lane; one sequence per CTA (up to 592) and eight."""
    hp = Hyper(cap_mode=cap_mode, L_max=256, smooth_radius=2)
    eng = _engine(hp, max_batch=1, max_window=W)
    r = np.random.default_rng(W + B)
    mask_id = WL.mask_id
    win = r.integers(1, W + 1, B).astype(np.int32)
    win[:2] = W
    remain = r.integers(1, 300, B).astype(np.int32)
    I = (np.abs(r.standard_normal((B, W))) * np.exp(-np.arange(W) / 16.0)).astype(np.float32)
    H = (r.random((B, W)) * 8).astype(np.float32)
    blk = np.array([r.integers(0, w + 1) for w in win]).astype(np.int32)
    conf = np.where(r.random((B, W)) < 0.5, 0.9 + 0.1 * r.random((B, W)), r.random((B, W))).astype(np.float32)
    x = (r.standard_normal((B, W, W)) * 6 - 12).astype(np.float32)
    ids = np.where(r.random((B, W)) < 0.8, mask_id, 5).astype(np.int32)
    dev = eng.device
    t = lambda a: torch.from_numpy(a).to(dev)
    f = lambda: torch.zeros((B, W), device=dev)
    bo = dict(score=f(), cum_influence=f(), cum_score=f(), block_len=torch.zeros((B,), dtype=torch.int32, device=dev))
    so = dict(sel_mask=torch.zeros((B, W), dtype=torch.uint8, device=dev),
              sel_idx=torch.zeros((B, W), dtype=torch.int32, device=dev),
              sel_count=torch.zeros((B,), dtype=torch.int32, device=dev))
    eng.boundary_batched(t(I), t(H), t(win), t(remain), bo)
    eng.select_batched(t(conf), t(ids), t(x), t(blk), t(win), so)
    eng.synchronize()
    g = {k: v.cpu().numpy() for k, v in {**bo, **so}.items()}
    for b in sorted({0, 1, B - 1} | set(r.integers(0, B, 20).tolist())):
        L, score, ci, cs = O.boundary(I[b], H[b], int(win[b]), int(remain[b]), True, _ocfg(hp))
        n = len(score)
        assert int(g["block_len"][b]) == L, b
        for name, want in (("score", score), ("cum_influence", ci), ("cum_score", cs)):
            assert np.array_equal(g[name][b, :n].view(np.uint32), want.view(np.uint32)), (b, name)
        w = int(win[b])
        want = O.cap_select(conf[b, :w], ids[b, :w] == mask_id, x[b, :w, :w], int(blk[b]), hp.tau_low, hp.tau_high,
                            hp.gamma, cap_mode)
        assert list(g["sel_idx"][b, :int(g["sel_count"][b])]) == want, b
        assert [i for i in range(w) if g["sel_mask"][b, i]] == want, b
    eng.close()


@pytest.mark.parametrize("cap_mode", [0, 1])
def test_select_with_nan_thresholds_as_the_comparisons_have_it(cap_mode):
    """No confidence is at or above a NaN, of either sign: no pool without tau_low (one token, the most confident),
    no first phase without tau_high."""
    eng = _engine(Hyper(cap_mode=cap_mode))
    r = np.random.default_rng(12)
    W, B = 100, 4
    conf = r.random((B, 128)).astype(np.float32)
    x = (r.standard_normal((B, 128, 128)) * 6 - 9).astype(np.float32)
    ids = np.full((B, 128), WL.mask_id, dtype=np.int32)
    nan = float("nan")
    for tl, th in ((nan, 0.95), (-nan, 0.95), (0.3, nan), (0.3, -nan), (nan, -nan)):
        g = eng.select(torch.from_numpy(ids).cuda(), [W] * B, conf=torch.from_numpy(conf).cuda(),
                       xlogp=torch.from_numpy(x).cuda(), block_len=torch.full((B,), W, dtype=torch.int32).cuda(),
                       thresholds=(tl, th, -8.0))
        eng.synchronize()
        for b in range(B):
            want = O.cap_select(conf[b, :W], ids[b, :W] == WL.mask_id, x[b, :W, :W], W, tl, th, -8.0, cap_mode)
            assert g["sel_idx"][b, :int(g["sel_count"][b])].tolist() == want, (tl, th, b)
    eng.close()


@pytest.mark.parametrize("cap_mode", [0, 1])
@pytest.mark.parametrize("W", [80, 128, 144, 256])
@pytest.mark.parametrize("conflicts", [0.0, 0.004, 0.05])
def test_select_long_greedy_passes_bit_exact(W, cap_mode, conflicts):
    """Pools of a hundred and more positions of which few or none conflict, ties among the confidences and decoded
    positions between them; every fourth sequence has a pool of just under or over what goes on in rank order."""
    hp = Hyper(tau_low=0.5, tau_high=0.9, cap_mode=cap_mode)
    eng = _engine(hp, max_batch=1, max_window=W)
    r = np.random.default_rng(W + cap_mode)
    B, mask_id = 12, WL.mask_id
    conf = (0.5 + 0.5 * r.random((B, W))).astype(np.float32)
    conf[:, ::5] = np.float32(0.75)                                            # ties
    conf[1] = np.float32(0.6)
    conf[2::4, 30:] = np.float32(0.1)                                          # pools of some 27
    x = np.where(r.random((B, W, W)) < conflicts, 0.0, -30.0 - 4 * r.random((B, W, W))).astype(np.float32)
    shift = 1 if conflicts == 0.004 else 0      # (also from a buffer that does not start on a 16-byte boundary)
    ids = np.where(r.random((B, W)) < 0.9, mask_id, 5).astype(np.int32)
    ids[0] = mask_id
    win = np.where(np.arange(B) % 3 == 2, W - 7, W).astype(np.int32)
    dev = eng.device
    t = lambda a: torch.from_numpy(a).to(dev)
    xd = torch.empty(x.size + 4, device=dev)[shift:shift + x.size].view(x.shape).copy_(t(x))
    so = dict(sel_mask=torch.zeros((B, W), dtype=torch.uint8, device=dev),
              sel_idx=torch.zeros((B, W), dtype=torch.int32, device=dev),
              sel_count=torch.zeros((B,), dtype=torch.int32, device=dev))
    eng.select_batched(t(conf), t(ids), xd, t(win), t(win), so)
    eng.synchronize()
    for b in range(B):
        w = int(win[b])
        want = O.cap_select(conf[b, :w], ids[b, :w] == mask_id, x[b, :w, :w], w, hp.tau_low, hp.tau_high, hp.gamma, cap_mode)
        assert so["sel_idx"][b, :int(so["sel_count"][b])].tolist() == want, b
        assert so["sel_mask"][b, :w].nonzero().flatten().tolist() == want, b
    eng.close()


@pytest.mark.parametrize("mode,norm", [(0, 0), (0, 1), (1, 2), (1, 1)])
@pytest.mark.parametrize("radius", [0, 1, 3, 8])
@pytest.mark.parametrize("W,B", [(144, 24), (256, 24), (256, 4097)])
def test_boundary_of_wide_windows_bit_exact(W, B, mode, norm, radius):
    """Windows above 128: four warps a sequence up to 4096 sequences, one beyond; lengths that end in any warp."""
    hp = Hyper(boundary_mode=mode, norm_mode=norm, smooth_radius=radius, L_max=256)
    eng = _engine(hp, max_batch=1, max_window=W)
    r = np.random.default_rng(W + B + 7 * radius + norm)
    win = r.integers(1, W + 1, B).astype(np.int32)
    win[:8] = [1, 2, 63, 64, 65, 128, 129, W]
    remain = r.integers(200, 300, B).astype(np.int32)
    have = (r.random(B) < 0.9).astype(np.int32)
    I = (np.abs(r.standard_normal((B, W))) * np.exp(-np.arange(W) / 60.0)).astype(np.float32)
    H = (r.random((B, W)) * r.uniform(0.01, 1.0, (B, 1))).astype(np.float32)   # boundaries far out, too
    dev = eng.device
    t = lambda a: torch.from_numpy(a).to(dev)
    f = lambda: torch.zeros((B, W), device=dev)
    bo = dict(score=f(), cum_influence=f(), cum_score=f(), block_len=torch.zeros((B,), dtype=torch.int32, device=dev))
    eng.boundary_batched(t(I), t(H), t(win), t(remain), bo, have_prev=t(have))
    eng.synchronize()
    g = {k: v.cpu().numpy() for k, v in bo.items()}
    for b in list(range(24)) + [B - 1]:
        L, score, ci, cs = O.boundary(I[b], H[b], int(win[b]), int(remain[b]), bool(have[b]), _ocfg(hp))
        n = len(score)
        assert int(g["block_len"][b]) == L, b
        for name, want in (("score", score), ("cum_influence", ci), ("cum_score", cs)):
            assert np.array_equal(g[name][b, :n].view(np.uint32), want.view(np.uint32)), (b, name)
        assert not g["score"][b, n:].any()
    eng.close()
