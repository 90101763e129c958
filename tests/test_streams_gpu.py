"""Two contexts on two streams, their launches interleaved from one thread: each gives
what it gives alone (the launches share SMs, shared memory and tensor memory)."""
import pytest
import torch

from paper_2505_14260_gb300 import msd, synth
from tests.gpu_support import open_engine

pytestmark = pytest.mark.gpu

TINY = synth.WORKLOADS["tiny"]


def _program(wl, rows, k, o, seed):
    """A generator of one context's work on the stream it is given: a prompt, a product of
    the caller's own weight (65 to 128 rows: CTAs that take an SM's whole tensor memory),
    steps as calls and as replayed graphs. Returns its results through `out`."""
    eng, _ = open_engine(wl.with_(seed=seed), steps=8)
    prompt = msd.upload_prompts(synth.make_prompts(wl.with_(seed=seed)))
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.bfloat16 if wl.dtype == "bf16" else torch.float32
    x = torch.randn(rows, k, generator=g, device="cuda").to(dt)
    w = torch.randn(o, k, generator=g, device="cuda").to(dt)
    y = torch.zeros(rows, o, device="cuda")
    torch.cuda.synchronize()

    def run(stream, out):
        eng.prefill(*prompt, stream=stream)
        yield
        for i in range(8):
            eng.linear(x, w, y, accumulate=i > 0, stream=stream)
            yield
            (eng.step if i % 2 else eng.step_calls)(stream=stream)
            yield
        out += [y, eng.tree.tokens, eng.argmax, eng.state()["seq_len"], eng.state()["target_kv"]]
    return eng, run


@pytest.mark.parametrize("a,b", [
    (TINY.with_(dtype="bf16"), TINY.with_(dtype="bf16", tree_nodes=70, topk=8)),
    (TINY.with_(dtype="bf16", hidden=512, n_heads=4, head_dim=128, ffn=1376, tree_nodes=60, topk=8),
     TINY.with_(dtype="bf16", batch=4, n_vis=(64, 150))),
    (TINY, TINY.with_(dtype="bf16", tree_nodes=40, topk=8)),
])
def test_two_contexts_on_two_streams(a, b):
    programs = [_program(a, 72, 2048, 1536, 11), _program(b, 80, 4096, 640, 12)]
    alone, together = [], []
    for eng, run in programs:
        out = []
        for _ in run(torch.cuda.Stream(), out):
            pass
        torch.cuda.synchronize()
        alone.append([t.clone() for t in out])
    outs, live = [[], []], []
    for (eng, run), out in zip(programs, outs):
        live.append(run(torch.cuda.Stream(), out))
    while live:
        live = [r for r in live if next(r, live) is not live]
    torch.cuda.synchronize()
    together = [[t.clone() for t in out] for out in outs]
    for one, two in zip(alone, together):
        for t, u in zip(one, two):
            assert torch.equal(t, u)
    for eng, _ in programs:
        eng.close()
