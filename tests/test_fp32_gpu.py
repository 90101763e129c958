"""The fp32 kernels at the edges of their tiles: the CUDA-core GEMM against
float64 products, and the attention (row tiles of 16 and 64, key splits, tree
tiles, both head dims) through whole steps against the oracle."""
import numpy as np
import pytest
import torch

from paper_2505_14260_gb300 import msd, synth
from tests.gpu_support import open_engine, record_buffers
from tests.parity_support import run_parity

pytestmark = pytest.mark.gpu

TINY = synth.WORKLOADS["tiny"]

# (m, k, o, x row padding, x offset in elements): tile edges of the 16-, 32- and
# 64-row tiles, K below, at and past a 64-k stage and over several K splits,
# rows and pointers that are not 16-byte aligned
GEMM = [(1, 1, 1, 0, 0), (1, 64, 33, 0, 0), (16, 256, 256, 0, 0), (17, 260, 65, 4, 0), (32, 2816, 64, 0, 0),
        (33, 127, 129, 0, 0), (64, 8192, 16, 0, 0), (65, 66, 700, 1, 0), (5, 4096, 1024, 0, 1),
        (200, 1028, 500, 0, 0), (7, 3, 2000, 2, 3)]
# every tile and split of the rule: 24-row tiles (one and several, short last ones), 128-row
# tiles with short last rows and columns, two and four splits
GEMM += [(24, 1024, 4000, 0, 0), (24, 2816, 1024, 4, 0), (20, 200, 5000, 1, 0), (48, 130, 3000, 0, 0),
         (100, 512, 5632, 0, 0), (341, 256, 5632, 0, 0), (341, 2816, 1024, 0, 0), (700, 129, 2900, 0, 1),
         (1500, 64, 3072, 0, 0), (257, 60, 6000, 3, 2), (16, 1024, 1024, 0, 0)]


@pytest.mark.parametrize("m,k,o,pad,off", GEMM)
@pytest.mark.parametrize("accumulate", [False, True])
def test_fp32_linear_matches_float64(m, k, o, pad, off, accumulate):
    eng, _ = open_engine(TINY, steps=1)
    g = torch.Generator(device="cuda").manual_seed(m * 7 + k * 3 + o)
    buf = torch.randn(off + m * (k + pad), generator=g, device="cuda")
    x = buf[off:].view(m, k + pad)[:, :k]
    w = torch.randn(o, k, generator=g, device="cuda")
    y = torch.randn(m, o, generator=g, device="cuda")
    ref = x.double() @ w.double().T + (y.double() if accumulate else 0.0)
    mag = x.double().abs() @ w.double().abs().T + (y.double().abs() if accumulate else 0.0)
    st = msd.lib().msd_linear(eng.ctx, x.data_ptr(), k + pad, m, k, w.data_ptr(), o, y.data_ptr(), o,
                              int(accumulate), 0)
    assert st == msd.MSD_OK
    torch.cuda.synchronize()
    # any order of k fp32 products and sums: (k + 1) rounding errors of 2^-24
    assert bool(((y.double() - ref).abs() <= (k + 1) * 2.0 ** -24 * mag + 1e-30).all())
    eng.close()


# more rows than the grid's 65535 row tiles of 24, and the most that 65535 of 64 hold
@pytest.mark.parametrize("m,o", [(65535 * 24 + 1, 8), (65535 * 64, 3), (65535 * 32 + 5, 80)])
def test_fp32_linear_takes_many_rows(m, o):
    eng, _ = open_engine(TINY, steps=1)
    g = torch.Generator(device="cuda").manual_seed(o)
    x = torch.randn(m, 4, generator=g, device="cuda")
    w = torch.randn(o, 4, generator=g, device="cuda")
    y = torch.full((m, o), float("nan"), device="cuda")
    eng.linear(x, w, y)
    ref = x.double() @ w.double().T
    assert bool(((y.double() - ref).abs() <= 5 * 2.0 ** -24 * (x.double().abs() @ w.double().abs().T) + 1e-30).all())
    eng.close()


# N over the 16-row tiles (one, two, a remainder) and the 64-row ones, prefixes
# below a key tile, at its edge, past it, and over every split; hd 64 and 128
@pytest.mark.parametrize("hd,nodes,vis,text", [(64, 7, 0, 9), (64, 33, 100, 28), (64, 70, 600, 41),
                                               (128, 16, 30, 34), (128, 31, 700, 69), (128, 65, 64, 64)])
def test_fp32_steps_match_oracle(hd, nodes, vis, text):
    wl = TINY.with_(n_heads=256 // hd, head_dim=hd, tree_nodes=nodes, tree_depth=4, topk=5, n_vis=(vis,),
                    n_text=(text, text))
    run_parity(wl, 2, None)


def test_fp32_ragged_batch_matches_oracle():
    wl = TINY.with_(batch=3, n_vis=(8, 150), n_text=(5, 90), tree_nodes=20)
    run_parity(wl, 2, None)


def test_fp32_linear_rows_do_not_depend_on_each_other():
    """A row of X alone gives the values it gives among others of the same tile
    count (fixed summation order)."""
    eng, _ = open_engine(TINY, steps=1)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(48, 512, generator=g, device="cuda")
    w = torch.randn(300, 512, generator=g, device="cuda")
    y = torch.zeros(48, 300, device="cuda")
    eng.linear(x, w, y)
    x2 = torch.randn(48, 512, generator=g, device="cuda")
    x2[17] = x[17]
    y2 = torch.zeros(48, 300, device="cuda")
    eng.linear(x2, w, y2)
    assert np.array_equal(y[17].cpu().numpy(), y2[17].cpu().numpy())
    eng.close()


# A key that a row does not see takes no part in that row's attention, whatever its K/V
# hold: a NaN or an infinity stays with the rows that see it. (The prompts run over
# several row and key tiles and, with few rows, over several key splits.)
NONFINITE = [float("nan"), float("inf")]


def _prompt(wl, bad=None, at=0):
    p = synth.make_prompts(wl)[0]
    if bad is not None:
        p.vis[at] = bad
    return msd.upload_prompts([p])


@pytest.mark.parametrize("bad", NONFINITE)
@pytest.mark.parametrize("hd,vis,at", [(64, 40, 30), (64, 200, 70), (128, 100, 60), (128, 700, 555)])
def test_fp32_prefill_rows_before_a_nonfinite_one(hd, vis, at, bad):
    wl = TINY.with_(n_heads=256 // hd, head_dim=hd, n_vis=(vis,), n_text=(30, 30), n_sys=8)
    eng, _ = open_engine(wl, steps=1)
    kv = []
    for b in (None, bad):
        eng.prefill(*_prompt(wl, b, at))
        s = eng.state()
        kv.append((s["target_kv"].clone(), s["draft_kv"].clone()))
    pos = 8 + at                            # the row's position (the draft row before it holds its embedding)
    assert torch.isnan(kv[1][0][-1, :, 0, :, pos]).all()
    for c, n in ((0, pos), (1, pos - 1)):
        assert torch.equal(kv[0][c][..., :n, :], kv[1][c][..., :n, :])
    eng.close()


@pytest.mark.parametrize("bad", NONFINITE)
@pytest.mark.parametrize("hd,nodes,vis", [(64, 16, 64), (64, 70, 300), (128, 33, 500)])
def test_fp32_verify_siblings_of_a_nonfinite_node(hd, nodes, vis, bad):
    wl = TINY.with_(n_heads=256 // hd, head_dim=hd, tree_nodes=nodes, topk=8, n_vis=(vis,))
    eng, w = open_engine(wl, steps=1)
    prompt = _prompt(wl)
    root = int(eng.prefill(*prompt)[0])
    used = set(prompt[0][0].tolist()) | {root}
    toks = [t for t in range(wl.vocab) if t not in used][:nodes]
    bad_tok, toks[0] = toks[0], root
    parent = [-1] + [(i - 1) // 3 for i in range(1, nodes)]
    under = {2}                             # node 2 and what hangs below it
    for i in range(3, nodes):
        if parent[i] in under:
            under.add(i)
    eng.w["embed"][bad_tok] = bad
    out = []
    for t2 in (toks[2], bad_tok):
        logits = torch.zeros(nodes, wl.vocab, device="cuda")
        eng.plant(eng.tree, 0, toks[:2] + [t2] + toks[3:], parent)
        eng.verify(logits=logits)
        out.append(logits)
    keep = [i for i in range(nodes) if i not in under]
    assert torch.isnan(out[1][2]).all() and not torch.isnan(out[0]).any()
    assert torch.equal(out[0][keep], out[1][keep])
    eng.close()


def test_fp32_draft_after_a_nonfinite_prompt():
    """Slots of the draft tree that a pass has not written yet hold the last tree's values."""
    wl = TINY.with_(n_sys=8, tree_nodes=40, tree_depth=5, topk=6)
    recs = []
    for first in (None, float("nan")):
        eng, w = open_engine(wl, steps=1)
        if first is not None:
            eng.prefill(*_prompt(wl, first, 20))
            eng.draft_tree()
        eng.prefill(*_prompt(wl))
        rec = record_buffers(wl)
        eng.draft_tree(record=rec)
        torch.cuda.synchronize()
        recs.append((rec["logits"].cpu(), eng.tree.tokens.cpu(), eng.tree.parent.cpu()))
        eng.close()
    assert not torch.isnan(recs[0][0]).any()
    assert all(torch.equal(a, b) for a, b in zip(*recs))


def test_fp32_one_row_of_very_many_requests():
    """Plain decoding of more requests than 15/16 of the grid's 65535 row tiles."""
    wl = TINY.with_(n_layers=1, hidden=64, n_heads=1, ffn=64, vocab=64, tree_nodes=1, tree_depth=1, topk=1,
                    n_vis=(0,), n_text=(2, 2), steps=2)
    g = torch.Generator().manual_seed(1)
    ids = torch.randint(0, 64, (62000, 2), generator=g, dtype=torch.int32).cuda()
    out = []
    for b in (62000, 5):
        eng, _ = open_engine(wl, steps=2, batch=b)
        eng.prefill(ids[:b].contiguous(), [2] * b, None, [0] * b)
        out.append([eng.ar_step().clone() for _ in range(2)])
        torch.cuda.synchronize()
        eng.ar_step()
        eng.close()
    for many, few in zip(*out):
        assert torch.equal(many[:5], few)
