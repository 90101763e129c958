"""The two-SM persistent GEMM (more than 128 token rows) at the edges of its
tiles: an odd count of 128-row weight tiles, a last tile with few rows, token
tiles of every width class, one K-block, ragged K, few and many pieces."""
import pytest
import torch

from paper_2505_14260_gb300 import synth
from tests.gpu_support import open_engine
from tests.parity_support import run_parity

pytestmark = pytest.mark.gpu

SHAPES = [(129, 64, 128), (129, 8, 1), (144, 72, 300), (255, 4096, 129), (256, 256, 384), (257, 2048, 256),
          (640, 4096, 640), (961, 200, 2000), (1025, 1024, 4096), (333, 11008, 128), (2000, 136, 72)]


@pytest.mark.parametrize("m,k,o", SHAPES)
def test_linear_many_rows(m, k, o):
    eng, _ = open_engine(synth.WORKLOADS["tiny"].with_(dtype="bf16"), steps=1)
    g = torch.Generator(device="cuda").manual_seed(m + k + o)
    x = torch.randn(m, k, generator=g, device="cuda").bfloat16()
    w = torch.randn(o, k, generator=g, device="cuda").bfloat16()
    y = torch.randn(m, o, generator=g, device="cuda")
    y0 = y.clone()
    ref = x.double() @ w.double().T
    mag = x.double().abs() @ w.double().abs().T
    for acc in (False, True, True):
        eng.linear(x, w, y, accumulate=acc)
    torch.cuda.synchronize()
    # exact products; every fp32 sum of up to k terms may truncate at 2^-23 of the
    # magnitudes summed, three times over
    assert bool(((y.double() - 3 * ref).abs() <= 3 * (k / 16 + 4) * 2.0 ** -23 * mag + 1e-6).all())
    y2 = y0.clone()
    eng.linear(x, w, y2)
    eng.linear(x, w, y0)
    assert torch.equal(y2, y0)                # deterministic
    eng.close()


# prompts longer than 128 rows through every projection (split operands, SwiGLU
# epilogue, residual adds): odd weight-tile counts (hidden 320, ffn 208), several chunks
@pytest.mark.parametrize("hidden,heads,ffn,vis,text", [(320, 5, 208, 120, 30), (256, 4, 688, 1000, 77),
                                                       (384, 3, 1040, 200, 57)])
def test_prefill_many_rows_matches_oracle(hidden, heads, ffn, vis, text):
    wl = synth.WORKLOADS["tiny"].with_(dtype="bf16", hidden=hidden, n_heads=heads, head_dim=hidden // heads, ffn=ffn,
                                       n_vis=(vis,), n_text=(text, text))
    run_parity(wl, 1, None)
