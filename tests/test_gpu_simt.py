"""CUDA-core kernels at the shapes where their tiles can go wrong, against the oracle."""
import pytest

from paper_2604_15750_b200 import inputs

from parity import Case, compare

pytestmark = pytest.mark.gpu


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
    gpu, ora = case.run_gpu(eng, poison=True), case.run_oracle()
    compare(case, gpu, ora)
    eng.set_option(1, 0)                       # DC_OPT_COOPERATIVE off: one launch per operation
    one = case.run_gpu(eng, poison=True)
    tol = 1e-5 if wl.dtype == "f32" else 2e-2
    for b in range(wl.batch):
        n = lengths["win_len"][b]
        for k in ("conf", "entropy", "lse"):
            assert abs(gpu[k][b, :n] - one[k][b, :n]).max() <= tol * max(1.0, abs(one[k][b, :n]).max()), (k, b)
    eng.close()
