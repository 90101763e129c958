"""The tensor-core GEMMs on the caller's row-major weights, through both entry
points, at the edges of their tiles: the two-SM persistent kernel (more than 128
token rows: an odd count of 128-row weight tiles, a last tile with few rows,
token tiles of every width class, one K-block, ragged K, few and many pieces)
and the cluster kernel (up to 128 rows, every K split); and prompts through the
packed weights."""
import ctypes

import pytest
import torch

from paper_2505_14260_gb300 import msd, synth
from tests.gpu_support import open_engine
from tests.parity_support import run_parity

pytestmark = pytest.mark.gpu

SHAPES = [(129, 64, 128), (129, 8, 1), (144, 72, 300), (255, 4096, 129), (256, 256, 384), (257, 2048, 256),
          (640, 4096, 640), (961, 200, 2000), (1025, 1024, 4096), (333, 11008, 128), (2000, 136, 72)]


SHAPES += [(1, 8, 1), (7, 4096, 129), (16, 2048, 40000), (17, 72, 1000), (33, 11008, 64), (60, 4096, 4096),
           (128, 1032, 500), (100, 64, 20000)]
# narrow tiles with up to 16 accumulators, cut short-K tiles, one CTA per SM past 64 rows
SHAPES += [(349, 944, 216), (309, 456, 77), (1309, 7184, 68), (176, 11008, 4096), (129, 4096, 1000),
           (119, 1520, 126), (80, 400, 300), (60, 304, 121), (7, 536, 19502)]


@pytest.mark.parametrize("m,k,o", SHAPES)
def test_linear_matches_float64(m, k, o):
    eng, _ = open_engine(synth.WORKLOADS["tiny"].with_(dtype="bf16"), steps=1)
    g = torch.Generator(device="cuda").manual_seed(m + k + o)
    x = torch.randn(m, k + 8, generator=g, device="cuda").bfloat16()[:, :k]      # rows with a stride
    w = torch.randn(o, k, generator=g, device="cuda").bfloat16()
    y = torch.randn(m, o, generator=g, device="cuda")
    y0 = y.clone()
    yn = torch.full((m, o + 3), 7.0, device="cuda")
    ref = x.double() @ w.double().T
    mag = x.double().abs() @ w.double().abs().T
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for acc in (False, True, True):
        eng.linear(x, w, y, accumulate=acc)
        assert msd.lib().msd_linear_noalloc(x.data_ptr(), k + 8, m, k, w.data_ptr(), o, yn.data_ptr(), o + 3,
                                            int(acc), stream) == msd.MSD_OK
    torch.cuda.synchronize()
    # exact products; every fp32 sum of up to k terms may truncate at 2^-23 of the
    # magnitudes summed, three times over
    bound = 3 * (k / 16 + 8) * 2.0 ** -23 * mag + 1e-6
    assert bool(((y.double() - 3 * ref).abs() <= bound).all())
    assert bool(((yn[:, :o].double() - 3 * ref).abs() <= bound).all())
    assert bool((yn[:, o:] == 7.0).all())     # nothing is written past a row's outputs
    y2 = y0.clone()
    eng.linear(x, w, y2)
    eng.linear(x, w, y0)
    assert torch.equal(y2, y0)                # deterministic
    eng.close()


# (m, k, o, chunks of a whole tile, cut tiles): whole tiles in chunks, cut tiles beside
# them, cut tiles alone, and products whose pieces would be too long; cluster shapes of
# 65 to 128 rows whose CTAs hold 512 columns, and the longest chain of the rule
CHAINS = [(131, 1560, 20225, 2, 0), (700, 4096, 11000, 3, 0), (264, 4208, 9927, 3, 2), (275, 3352, 19573, 3, 0),
          (500, 11008, 14336, 8, 0), (1953, 15728, 259, 0, 36), (72, 11008, 9472, 1, 0), (65, 8192, 1001, 1, 0),
          (80, 11008, 500, 1, 0), (128, 11008, 20000, 1, 0)]


@pytest.mark.parametrize("accumulate", [False, True])
@pytest.mark.parametrize("m,k,o,chunks,cut", CHAINS)
def test_linear_error_follows_the_chains(m, k, o, chunks, cut, accumulate):
    """The accumulators truncate: a step of 16 terms loses half a unit in the last place on
    average, at most 2^-24 of the partial sum, which grows like the square root of the
    terms (2/3 of the result on average). Four steps a K-block over the launch's longest
    chain bound every output column's error; the sums of accumulators, pieces and chunks
    and the residual round once each (2^-24, some ten of them)."""
    shape = msd.msd_gemm_shape()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert msd.lib().msd_test_gemm_shape(m, k, o, 1, 0, sms, ctypes.byref(shape)) == msd.MSD_OK
    if sms == 152:
        assert (shape.chunks, shape.cut_tiles) == (chunks, cut)
    eng, _ = open_engine(synth.WORKLOADS["tiny"].with_(dtype="bf16"), steps=1)
    g = torch.Generator(device="cuda").manual_seed(m + k + o)
    x = torch.randn(m, k, generator=g, device="cuda").bfloat16()
    w = torch.randn(o, k, generator=g, device="cuda").bfloat16()
    y = torch.randn(m, o, generator=g, device="cuda") if accumulate else torch.full((m, o), float("nan"), device="cuda")
    yn = y.clone()
    ref = x.double() @ w.double().T
    if accumulate:
        ref += y
    eng.linear(x, w, y, accumulate=accumulate)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert msd.lib().msd_linear_noalloc(x.data_ptr(), k, m, k, w.data_ptr(), o, yn.data_ptr(), o, int(accumulate),
                                        stream) == msd.MSD_OK
    bound = 4 * shape.chain * 2.0 ** -24 * 2 / 3 + 10 * 2.0 ** -24
    for out in (y, yn):         # (the scratch of the second call may cut fewer tiles: no longer chains)
        err = (out.double() - ref).norm(dim=0) / ref.norm(dim=0)
        assert float(err.max()) <= bound, (float(err.max()), bound)
    eng.close()


def test_linear_reads_a_weight_written_just_before():
    """The weight and the rows come from kernels launched right before the call."""
    eng, _ = open_engine(synth.WORKLOADS["tiny"].with_(dtype="bf16"), steps=1)
    for m in (16, 300):
        x = torch.zeros(m, 1024, device="cuda").bfloat16()
        w = torch.zeros(2048, 1024, device="cuda").bfloat16()
        y = torch.zeros(m, 2048, device="cuda")
        for i in range(1, 6):
            x.fill_(float(i))
            w.fill_(0.5)
            eng.linear(x, w, y)
            assert bool((y == 512.0 * i).all()), (m, i)
    eng.close()


def test_linear_refuses_unaligned_operands():
    eng, _ = open_engine(synth.WORKLOADS["tiny"].with_(dtype="bf16"), steps=1)
    buf = torch.zeros(4096, device="cuda").bfloat16()
    y = torch.zeros(4, 4, device="cuda")
    st = msd.lib().msd_linear(eng.ctx, buf.data_ptr() + 2, 16, 4, 16, buf.data_ptr(), 4, y.data_ptr(), 4, 0, 0)
    assert st == msd.MSD_ERR_INVALID
    st = msd.lib().msd_linear_noalloc(buf.data_ptr(), 16, 4, 16, buf.data_ptr() + 2, 4, y.data_ptr(), 4, 0, 0)
    assert st == msd.MSD_ERR_INVALID
    eng.close()


# prompts longer than 128 rows through every projection (split operands, SwiGLU
# epilogue, residual adds): odd weight-tile counts (hidden 320, ffn 208), several chunks
@pytest.mark.parametrize("hidden,heads,ffn,vis,text", [(320, 5, 208, 120, 30), (256, 4, 688, 1000, 77),
                                                       (384, 3, 1040, 200, 57)])
def test_prefill_many_rows_matches_oracle(hidden, heads, ffn, vis, text):
    wl = synth.WORKLOADS["tiny"].with_(dtype="bf16", hidden=hidden, n_heads=heads, head_dim=hidden // heads, ffn=ffn,
                                       n_vis=(vis,), n_text=(text, text))
    run_parity(wl, 1, None)
