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
