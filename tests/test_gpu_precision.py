"""What the launch-per-GEMM path (more than 256 activation rows) holds and sums in 32 bits, seen through bf16 outputs:
results that cancel show an error of 1e-6 of their terms, which the rounding of a full-size result hides."""
import math

import numpy as np
import pytest
import torch

from paper_2604_15750_b200 import DepCap

pytestmark = pytest.mark.gpu
DEV, BF16 = "cuda", torch.bfloat16


def _prefill(layers, embed_row, n_q, n_kv, d, ff, tokens, theta=10000.0):
    """K and V rows that a prompt of `tokens` equal tokens leaves: [layers, n_kv, tokens, 128] and [.., 128, tokens]."""
    lw = [dict(dict(wq=torch.zeros(n_q * 128, d), wk=torch.zeros(n_kv * 128, d), wv=torch.zeros(n_kv * 128, d),
                    wo=torch.zeros(d, n_q * 128), w_gate=torch.zeros(ff, d), w_up=torch.zeros(ff, d),
                    w_down=torch.zeros(d, ff), norm1=torch.ones(d), norm2=torch.ones(d)), **l) for l in layers]
    dev = lambda t: t.to(BF16).to(DEV).contiguous()
    weights = dict(embed=dev(embed_row.expand(64, d)), lm_head=dev(torch.zeros(64, d)), final_norm=dev(torch.ones(d)),
                   layers=[{k: dev(v) for k, v in l.items()} for l in lw])
    ctx = (tokens + 63) // 64 * 64
    eng = DepCap(n_layers=len(layers), d_model=d, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=128, d_ff=ff, vocab=64, mask_id=63,
                 dtype="bf16", weights=weights, max_batch=1, max_ctx=ctx, max_last=tokens, max_window=16, rope_theta=theta)
    kc = torch.zeros((len(layers), 1, n_kv, ctx, 128), dtype=BF16, device=DEV)
    vc = torch.zeros((len(layers), 1, n_kv, 128, ctx), dtype=BF16, device=DEV)
    st = eng.prefill(kc, vc, torch.ones((1, tokens), dtype=torch.int32, device=DEV), [tokens])
    eng.synchronize()
    assert int(st[0]) == 0
    eng.close()
    return kc[:, 0, :, :tokens].double().cpu().numpy(), vc[:, 0, :, :, :tokens].double().cpu().numpy()


def test_rotated_keys_have_the_tables_precision():
    """All rows norm to ones and one weight a feature: the keys in front of the rotation are the weights a, b of a
    pair.  The factors are fp32, rounded once (2^-25 each), a product is rounded (2^-24 of it) and so is the sum: 2^-23 of
    |a| + |b| covers them.  Half a million pairs, all of high frequency, have results near zero, where the
    rounding to bf16 hides nothing of that size."""
    n, nkv, d, theta = 1008, 8, 256, 2.0
    g = torch.Generator().manual_seed(5)
    w = (0.5 + torch.rand(nkv, 128, generator=g)).to(BF16).double()
    wk = torch.zeros(nkv * 128, d)
    wk[:, 0] = w.reshape(-1).float()
    got, _ = _prefill([dict(wk=wk)], torch.ones(d), nkv, nkv, d, 256, n, theta)
    ang = np.arange(n)[:, None] * theta ** (-2.0 * np.arange(64) / 128.0)
    c, s = np.cos(ang), np.sin(ang)
    a, b = (x[:, None, :].numpy() for x in (w[:, :64], w[:, 64:]))
    ref = np.concatenate([a * c - b * s, b * c + a * s], -1)
    terms = np.concatenate([a + b] * 2, -1)
    half_ulp = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(got[0]), np.abs(ref)))) - 8)
    over = ((np.abs(got[0] - ref) - half_ulp) / terms).max()
    print("largest error past the rounding to bf16, of the terms:", over)
    assert over <= 2.0 ** -23


def _cancelling(rows, K, g):
    """[rows, K] bf16 numbers: random positive ones whose sum the last 64 take back, exactly."""
    w = (0.5 + torch.rand(rows, K, generator=g)).to(BF16).double()
    left = w[:, :K - 64].sum(1)
    for k in range(K - 64, K):
        take = left / max(K - 8 - k, 1)
        w[:, k] = (-take).to(BF16).double()
        left = left + w[:, k]
    return w


@pytest.mark.parametrize("where", ["qkv", "down"])
def test_sums_are_taken_in_chains_as_short_as_the_fused_chains(where):
    """The tensor cores truncate a running fp32 sum at every MMA, so its error grows with the MMAs of one
    accumulator.  The same sums on both paths, 256 rows (two accumulators a GEMM, and K splits) and 1024 rows: the error
    of the second may not be larger (a factor 1.25 for other orders; one accumulator over all k shows 4)."""
    err = {}
    for tokens in (256, 1024):
        g = torch.Generator().manual_seed(7)
        if where == "qkv":
            # a gain of 171 / 128: the products have 16 bits, their sums more than 24; 128 tiles of 128 features for the
            # fused chain, too many for it to hand a part of k to other CTAs, 36 for the other path, a unit a worker
            d, nq, nkv = (4096, 64, 32) if tokens == 256 else (4096, 28, 4)
            w = _cancelling(256, d, g)
            wv = torch.zeros(nkv * 128, d)
            wv[:256] = w.float()
            _, v = _prefill([dict(wv=wv, norm1=torch.full((d,), 171 / 128))], torch.ones(d), nq, nkv, d, 256, tokens)
            out, ref = v[0][:2].reshape(256, tokens)[:, 0], w.sum(1).numpy()
        else:
            # x = (1, 0, ..): the norm gives 32 in feature 0, gate and up make the activations equal; the down projection
            # of layer 0 adds cancelling sums to x, whose norm (32 of them) layer 1 hands on as its values
            d, ff = 1024, 8192
            gate, up, pick = torch.zeros(ff, d), torch.zeros(ff, d), torch.zeros(256, d)
            gate[:, 0] = 4.0 / 32
            up[:, 0] = 0.25451 / 32          # 1 / silu(4)
            pick[torch.arange(256), torch.arange(256) + 1] = 1.0
            w = _cancelling(d, ff, g)
            w[0] = 0
            emb = torch.zeros(d)
            emb[0] = 1.0
            _, v = _prefill([dict(w_gate=gate, w_up=up, w_down=w.float()), dict(wv=pick)], emb, 2, 2, d, ff, tokens)
            out, ref = v[1].reshape(256, tokens)[:, 0] / 32, w[1:257].sum(1).numpy()
        err[tokens] = math.sqrt(((out - ref) ** 2).mean()) / w[:257].abs().sum(1).max().item()
    print(where, err)
    assert 0 < err[256] < 1e-4
    assert err[1024] <= 1.25 * err[256]
