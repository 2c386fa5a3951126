"""The work whose speed is tracked: block-steps, prefills, the decision calls and a decoding loop.

Every case goes through the public binding (`DepCap.step` / `select` / `prefill` / `generate` /
`boundary_batched` / `select_batched`) at full depth: random-init weights N(0, 0.02) of the
backbones in `inputs.WORKLOADS`, seeded token ids, a seeded N(0, 1) context cache.  As in the
benchmark, a step gets shaped LM-head inputs (`h_final`), because random-init logits are flat and
the decisions would be degenerate; the stack's own result is returned beside the decisions (`h_out`
and, where a step appends the last block to the cache, the K / V rows it wrote).
"""
import math

import numpy as np
import torch

from paper_2604_15750_b200 import DepCap, inputs

DEV = "cuda"
# backbone shapes by the name of the workload they come from
MODELS = {n: inputs.WORKLOADS[n] for n in ("tiny_f32", "llada8b_b1", "dream7b_b4", "dream7b_b4_bias")}


def _step(name, model, mode, batch, ctx, last, win, ctx_spread=0, win_spread=0, decoded=0):
    return dict(name=name, kind="step", model=model, mode=mode, batch=batch, ctx=ctx, ctx_spread=ctx_spread,
                last=last, win=win, win_spread=win_spread, decoded=decoded)


def listed():
    return [
        # the smallest call: one step of the fp32 model, launches and latency only
        _step("tiny step fp32", "tiny_f32", "boundary", 1, 64, 16, 32),
        # the whole decoding loop on the same model: host scheduling, read-backs and small kernels
        dict(name="tiny generate fp32", kind="generate", model="tiny_f32", batch=1, ctx=64, gen=48),
        # a serving layer that decides for many requests in one call
        dict(name="decide 8192x128", kind="decide", batch=8192, win=128),
        # interactive decoding: the boundary step (both variants) that opens every block
        _step("llada boundary b1", "llada8b_b1", "boundary", 1, 512, 32, 64),
        # ... with p_prev carried over from the boundary step before it; odd sizes in mid-generation
        _step("llada carried b1", "llada8b_b1", "carried", 1, 713, 27, 57),
        # ... and the denoising steps inside a block of L_min positions, most forwards of a generation
        _step("llada denoise b1", "llada8b_b1", "denoise", 1, 619, 0, 8, decoded=3),
        # a batch of ragged requests: boundary step and denoising step
        _step("llada boundary b8", "llada8b_b1", "boundary", 8, 1024, 32, 128, ctx_spread=256),
        _step("llada denoise b8", "llada8b_b1", "denoise", 8, 1200, 0, 24, ctx_spread=300, win_spread=16, decoded=2),
        # grouped KV heads
        _step("dream boundary b4", "dream7b_b4", "boundary", 4, 768, 32, 64),
        # long contexts: attention over 16 x 4096 cached keys
        _step("llada boundary long b16", "llada8b_b1", "boundary", 16, 4096, 32, 128),
        # prompts: one of ordinary length, and a short one of odd length
        dict(name="llada prefill 1024", kind="prefill", model="llada8b_b1", batch=1, tokens=1024, spread=0),
        dict(name="dream prefill 187", kind="prefill", model="dream7b_b4", batch=1, tokens=187, spread=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: each kind about as often as among the listed ones."""
    kind = rng.choice(["tiny", "generate", "decide", "decide", "boundary", "boundary", "boundary", "carried",
                       "denoise", "denoise", "prefill", "prefill"])
    if kind == "tiny":
        return _drawn("tiny_f32", rng.choice(["boundary", "boundary", "denoise"]), rng.randint(1, 3), rng.randint(1, 192),
                      rng.randint(1, 32), rng.randint(8, 64), rng)
    if kind == "generate":
        return dict(kind="generate", model="tiny_f32", batch=rng.randint(1, 3), ctx=rng.randint(1, 128), gen=rng.randint(16, 64))
    if kind == "decide":
        return dict(kind="decide", batch=_log(rng, 64, 8192), win=rng.randint(1, 16) * 16)
    model = rng.choice(["llada8b_b1", "llada8b_b1", "dream7b_b4", "dream7b_b4_bias"])
    if kind == "prefill":
        batch = rng.choice([1, 1, 1, 2, 4])
        tokens = _log(rng, 32, 4096 // batch)
        return dict(kind="prefill", model=model, batch=batch, tokens=tokens, spread=rng.randint(0, tokens // 4) if batch > 1 else 0)
    batch = rng.choice([1, 1, 1, 2, 3, 4, 8, 16])
    ctx = _log(rng, 64, 4096)
    if kind == "denoise":
        return _drawn(model, "denoise", batch, ctx, 0, _log(rng, 8, 64), rng)
    return _drawn(model, kind, batch, ctx, rng.randint(8, 32), _log(rng, 24, 128), rng)


def _drawn(model, mode, batch, ctx, last, win, rng):
    c = _step("", model, mode, batch, ctx, 0 if mode == "denoise" else last, win,
              ctx_spread=rng.randint(0, ctx // 3) if batch > 1 else 0,
              win_spread=rng.randint(0, win // 4) if batch > 1 else 0,
              decoded=rng.randint(0, win // 2) if mode == "denoise" else 0)
    del c["name"]
    return c


# ---- sizes -----------------------------------------------------------------------------------
def _up(v, m):
    return (v + m - 1) // m * m


def _ragged(n, spread, batch, stride):
    """Lengths of a batch: from n down by up to `spread`, no two neighbours alike."""
    return [n - (b * stride) % (spread + 1) for b in range(batch)]


def _lengths(case):
    B = case["batch"]
    ctx = _ragged(case["ctx"], case["ctx_spread"], B, 37)
    win = _ragged(case["win"], case["win_spread"], B, 5)
    return ctx, [case["last"]] * B, win


# ---- inputs ----------------------------------------------------------------------------------
def _normal(g, shape, std, dtype):
    return torch.empty(shape, dtype=dtype, device=DEV).normal_(0.0, std, generator=g)


def _weights(w, g):
    d, hq, hkv, F, t = w.d_model, w.n_q_heads * w.head_dim, w.n_kv_heads * w.head_dim, w.d_ff, w.torch_dtype
    mats = dict(wq=(hq, d), wk=(hkv, d), wv=(hkv, d), wo=(d, hq), w_gate=(F, d), w_up=(F, d), w_down=(d, F))
    if w.qkv_bias:
        mats.update(bq=(hq,), bk=(hkv,), bv=(hkv,))
    # a residual stream that no single layer outweighs, as in a trained model: unit embeddings, and the
    # two projections back to it drawn smaller by sqrt(2 * layers), as such backbones are initialised
    # (with 0.02 everywhere, as the two-layer fp32 model has it, the first layer drowns the embeddings
    # and rounding noise grows with depth)
    deep = w.n_layers > 2
    back = 0.02 / math.sqrt(2.0 * w.n_layers) if deep else 0.02
    layers = []
    for _ in range(w.n_layers):
        lw = {n: _normal(g, s, 0.5 if len(s) == 1 else back if n in ("wo", "w_down") else 0.02, t) for n, s in mats.items()}
        lw.update(norm1=torch.ones(d, dtype=t, device=DEV), norm2=torch.ones(d, dtype=t, device=DEV))
        layers.append(lw)
    return dict(embed=_normal(g, (w.vocab, d), 1.0 if deep else 0.02, t), lm_head=_normal(g, (w.vocab, d), 0.02, t),
                final_norm=torch.ones(d, dtype=t, device=DEV), layers=layers)


def _engine(w, weights, batch, max_ctx, max_last, max_win):
    return DepCap(n_layers=w.n_layers, d_model=w.d_model, n_q_heads=w.n_q_heads, n_kv_heads=w.n_kv_heads,
                  head_dim=w.head_dim, d_ff=w.d_ff, vocab=w.vocab, mask_id=w.mask_id, dtype=w.dtype, weights=weights,
                  max_batch=batch, max_ctx=max_ctx, max_last=max_last, max_window=max_win, rms_eps=w.rms_eps,
                  rope_theta=w.rope_theta)


def _caches(w, g, batch, max_ctx, fill):
    k = (w.n_layers, batch, w.n_kv_heads, max_ctx, w.head_dim)
    v = (w.n_layers, batch, w.n_kv_heads, w.head_dim, max_ctx)
    if fill:
        return _normal(g, k, 1.0, w.torch_dtype), _normal(g, v, 1.0, w.torch_dtype)
    return torch.zeros(k, dtype=w.torch_dtype, device=DEV), torch.zeros(v, dtype=w.torch_dtype, device=DEV)


def _steering(w, g, lm_head, B, W):
    """LM-head inputs [B, 2, W, d] with targets whose probability falls with the distance from the
    frontier, some conflicting pairs, and a prev variant that knows less near the frontier (the
    profile "decay" of inputs.make_steering)."""
    k = torch.arange(W, device=DEV, dtype=torch.float32)
    rand = lambda *s: torch.rand(s, device=DEV, generator=g)
    tgt = torch.randint(0, w.vocab - 1, (B, W), device=DEV, generator=g)
    a = (math.log(w.vocab) - 4.0) + 10.0 * rand(B, W) * torch.exp(-k / 48.0)
    paired = (rand(B, W) < 0.25) & (a > math.log(w.vocab) + 2.0)
    partner = torch.clamp(k.long() + torch.randint(1, 5, (B, W), device=DEV, generator=g), max=W - 1)
    u = lm_head[tgt].float()
    u /= (u * u).sum(-1, keepdim=True)
    up = torch.gather(u, 1, partner[..., None].expand_as(u))
    rows = a[..., None] * (u + 0.75 * paired[..., None] * up)
    noise = _normal(g, rows.shape, 1e-3, torch.float32)
    damp = (1.0 - 0.6 * torch.exp(-k / 16.0))[:, None]
    return torch.stack([rows + noise, damp * rows + noise], 1).to(w.torch_dtype).contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return {"step": _prepare_step, "generate": _prepare_generate, "decide": _prepare_decide,
            "prefill": _prepare_prefill}[case["kind"]](case, g)


def _prepare_step(case, g):
    w, B, mode = MODELS[case["model"]], case["batch"], case["mode"]
    ctx, last, win = _lengths(case)
    maxw, maxl = _up(case["win"], 16), max(case["last"], 1)
    weights = _weights(w, g)
    eng = _engine(w, weights, B, _up(case["ctx"] + case["last"], 64), maxl, maxw)
    kc, vc = _caches(w, g, B, eng.max_ctx, True)
    ids = lambda *s: torch.randint(0, w.mask_id, s, device=DEV, generator=g, dtype=torch.int32)
    win_ids = torch.full((B, maxw), w.mask_id, dtype=torch.int32, device=DEV)
    if case["decoded"]:     # a step in mid-block: some positions already hold their tokens
        at = torch.rand((B, maxw), device=DEV, generator=g).argsort(1)[:, :case["decoded"]]
        win_ids.scatter_(1, at, ids(B, case["decoded"]))
    h_out = torch.zeros((B, maxw, w.d_model), dtype=w.torch_dtype, device=DEV)
    boundary = mode != "denoise"
    carried = None
    if mode == "carried":   # rows of the window before, which had moved on by one block
        carried = (_normal(g, h_out.shape, 1.0, w.torch_dtype), [max(n - case["last"], 0) for n in win])
    s = dict(kind="step", eng=eng, win_ids=win_ids, win=win, block_len=None,
             args=dict(k_cache=kc, v_cache=vc, ctx_len=ctx, last_ids=ids(B, maxl), last_len=last, win_ids=win_ids,
                       win_len=win, remain_len=[n + 64 for n in win], influence=mode == "boundary", boundary=boundary,
                       h_final=_steering(w, g, weights["lm_head"], B, maxw), export_kv=boundary, carried=carried,
                       h_out=h_out))
    names = ["pred_id", "conf", "entropy", "lse", "xlogp", "status"]
    if boundary:
        names += ["influence", "score", "cum_influence", "cum_score", "block_len"]
        s["kv"] = [c for b in range(B) for c in (kc[:, b, :, ctx[b]:ctx[b] + last[b], :], vc[:, b, :, :, ctx[b]:ctx[b] + last[b]])]
    else:
        s["kv"] = []
        s["block_len"] = torch.tensor(win, dtype=torch.int32, device=DEV)   # the block is the whole window
    s["names"] = names
    return s


def _prepare_generate(case, g):
    w, B = MODELS[case["model"]], case["batch"]
    weights = _weights(w, g)
    eng = _engine(w, weights, B, _up(case["ctx"] + case["gen"], 64), 64, 64)
    kc, vc = _caches(w, g, B, eng.max_ctx, True)
    return dict(kind="generate", eng=eng, kc=kc, vc=vc, ctx=[case["ctx"]] * B, gen=case["gen"])


def _prepare_prefill(case, g):
    w, B = MODELS[case["model"]], case["batch"]
    n = _ragged(case["tokens"], case["spread"], B, 37)
    eng = _engine(w, _weights(w, g), B, _up(case["tokens"], 64), case["tokens"], 16)
    kc, vc = _caches(w, g, B, eng.max_ctx, False)
    ids = torch.randint(0, w.mask_id, (B, case["tokens"]), device=DEV, generator=g, dtype=torch.int32)
    kv = [c for b in range(B) for c in (kc[:, b, :, :n[b], :], vc[:, b, :, :, :n[b]])]
    return dict(kind="prefill", eng=eng, args=(kc, vc, ids, n), kv=kv)


def _prepare_decide(case, g):
    """Signals of many sequences as steered steps give them: influence and entropy that fall and
    rise with the distance from the frontier, half of the positions confident."""
    B, W, w = case["batch"], case["win"], MODELS["tiny_f32"]
    eng = _decider(W)
    rand = lambda *s: torch.rand(s, device=DEV, generator=g)
    k = torch.arange(W, device=DEV, dtype=torch.float32)
    infl = rand(B, W) * torch.exp(-k / 24.0)
    ent = rand(B, W) * (0.2 + k / W)
    sure = rand(B, W) < 0.5
    conf = torch.where(sure, 0.8 + 0.2 * rand(B, W), 0.8 * rand(B, W))
    xlogp = torch.rand((B, W, W), device=DEV, generator=g).mul_(-16.0).sub_(4.0)   # D = x_ij + x_ji around gamma - 8
    win_ids = torch.full((B, W), w.mask_id, dtype=torch.int32, device=DEV)
    win_ids[rand(B, W) < 0.15] = 5                                              # decoded already
    lens = dict(win_len=torch.randint(max(1, W // 2), W + 1, (B,), device=DEV, generator=g, dtype=torch.int32),
                remain=torch.randint(W, 4 * W + 1, (B,), device=DEV, generator=g, dtype=torch.int32),
                block=torch.randint(min(8, W), W + 1, (B,), device=DEV, generator=g, dtype=torch.int32))
    f = lambda: torch.zeros((B, W), dtype=torch.float32, device=DEV)
    i = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    return dict(kind="decide", eng=eng, infl=infl, ent=ent, conf=conf, xlogp=xlogp, win_ids=win_ids, lens=lens,
                bnd=dict(score=f(), cum_influence=f(), cum_score=f(), block_len=i(B)),
                sel=dict(sel_mask=torch.zeros((B, W), dtype=torch.uint8, device=DEV), sel_idx=i(B, W), sel_count=i(B)))


def _decider(W):
    """A context for the decision calls only: no layers, a small vocabulary."""
    w, g = MODELS["tiny_f32"], torch.Generator(device=DEV)
    g.manual_seed(1)
    weights = dict(embed=_normal(g, (w.vocab, w.d_model), 0.02, w.torch_dtype), layers=[],
                   lm_head=_normal(g, (w.vocab, w.d_model), 0.02, w.torch_dtype),
                   final_norm=torch.ones(w.d_model, dtype=w.torch_dtype, device=DEV))
    return DepCap(n_layers=0, d_model=w.d_model, n_q_heads=w.n_q_heads, n_kv_heads=w.n_kv_heads, head_dim=w.head_dim,
                  d_ff=w.d_ff, vocab=w.vocab, mask_id=w.mask_id, dtype=w.dtype, weights=weights, max_batch=1, max_ctx=0,
                  max_last=0, max_window=W)


# ---- one pass --------------------------------------------------------------------------------
def run(s):
    eng, kind = s["eng"], s["kind"]
    if kind == "step":
        out = eng.step(**s["args"])
        sel = eng.select(s["win_ids"], s["win"], block_len=s["block_len"])
        return [out[n] for n in s["names"]] + [sel["sel_mask"], sel["sel_count"], s["args"]["h_out"]] + s["kv"]
    if kind == "generate":
        tokens, blocks, nfe = eng.generate(s["kc"], s["vc"], s["ctx"], s["gen"])
        return [tokens, np.array([n for row in blocks for n in row], dtype=np.int32), nfe]
    if kind == "prefill":
        return [eng.prefill(*s["args"])] + s["kv"]
    lens = s["lens"]
    eng.boundary_batched(s["infl"], s["ent"], lens["win_len"], lens["remain"], s["bnd"])
    eng.select_batched(s["conf"], s["win_ids"], s["xlogp"], lens["block"], lens["win_len"], s["sel"])
    return [s["bnd"], s["sel"]]


# ---- what a pass cannot do without ---------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "decide":    # all rows once; of xlogp the rows and columns of the pool, about 0.42 of a block of 0.5 W
        B, W = case["batch"], case["win"]
        return dict(bytes=B * (4.0 * 4 * W + 4.0 * 3 * W + 5.0 * W + 4.0 * (0.42 * 0.5 * W) ** 2), flops=B * 60.0 * W)
    w = MODELS[case["model"]]
    es = 4 if w.dtype == "f32" else 2
    hq, hkv, d = w.n_q_heads * w.head_dim, w.n_kv_heads * w.head_dim, w.d_model
    layer = d * (2 * hq + 2 * hkv) + 3 * d * w.d_ff
    B = case["batch"]
    if kind == "generate":  # flat predictions: one token per forward, one sequence per weight pass at least
        rows = case["gen"] * 8.0 * B
        return dict(bytes=es * case["gen"] * (w.n_layers * layer + w.vocab * d), flops=2.0 * rows * (w.n_layers * layer + w.vocab * d))
    if kind == "prefill":
        n = _ragged(case["tokens"], case["spread"], B, 37)
        att = sum(4.0 * t * t * hq for t in n) * (w.n_layers - 1)
        # the last layer ends with its K / V projections
        used = (w.n_layers - 1) * layer + 2 * d * hkv
        return dict(bytes=es * (used + sum(n) * (d + 2.0 * w.n_layers * hkv)), flops=2.0 * sum(n) * used + att)
    ctx, last, win = _lengths(case)
    nv = 2 if case["mode"] == "boundary" else 1
    lv = 1 if case["mode"] == "denoise" else 2          # distributions per window position
    rows = [l + n for l, n in zip(last, win)]
    kv = sum(ctx) * 2 * hkv * w.n_layers
    att = sum(nv * 4.0 * r * (r + p) * hq for r, p in zip(rows, ctx)) * w.n_layers
    out = sum(4.0 * n * n + 40.0 * n + es * n * d * (1 + lv) for n in win) + (es * 2.0 * hkv * w.n_layers * sum(last))
    return dict(bytes=es * (w.n_layers * layer + w.vocab * d + kv + sum(rows) * d) + out,
                flops=2.0 * nv * sum(rows) * w.n_layers * layer + 2.0 * lv * sum(win) * w.vocab * d + att)


def tolerance(case):
    if case["kind"] == "decide":        # explicit roundings in a fixed order: a function of the input bits
        return "exact"
    if case["kind"] == "generate":      # tokens only
        return {"rel": 0.0, "differ": 0.005}
    if case["model"] == "tiny_f32":     # fp32 sums: 9e-7 (largest 2.3e-6) off the fp64 oracle
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.005}
    # bf16 at every GEMM input through 28 or 32 layers: the CUDA-core and the tensor-core kernels, which sum
    # in other orders, are 6e-3 (largest single value 3.6e-2) apart in h_out and the K / V rows
    return {"rel": 2.4e-2, "max": 0.15, "differ": 0.005}
