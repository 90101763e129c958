"""Performance cases of the MSD decode library: what a program that decodes with
it has it do, through the public binding (Engine and the C ABI).

Kinds of case
  draft_verify  msd_draft_tree (with its record) and msd_verify of the drafted
                tree, as separate calls: the loop of a program that looks at the
                tree and the logits of every step. Repeatable: neither call
                advances the sequence.
  prefill       msd_prefill of a batch of interleaved image + text prompts: the
                time to the first token. The caches are its result.
  verify        msd_verify of a caller-planted tree behind a prefilled prefix:
                one target forward, the bulk of every decode step.
  generate      a whole request: prefill, then replayed steps (greedy trees,
                sampling at T > 0, or plain greedy decoding), then the logits of a
                planted tree at the position reached.
  linear        one projection of the caller's own weight: msd_linear, or
                msd_linear_noalloc for callers without an allocator.

Models: the widths of this repository's workloads (tiny, 7B, 13B) and a
generic small one; layer counts are cut where a case stands for the layers and
not for a whole model. Random-init drafts are never accepted, so a step advances
by one token, as in the benchmark.
"""
import ctypes
import math
import random

import torch

from paper_2505_14260_gb300 import msd

TINY = dict(hidden=256, heads=4, ffn=688, vocab=1024)
SMALL = dict(hidden=1024, heads=16, ffn=2816, vocab=32000)      # a generic small decoder, head_dim 64
W7B = dict(hidden=4096, heads=32, ffn=11008, vocab=32000)
W13B = dict(hidden=5120, heads=40, ffn=13824, vocab=32000)
MODELS = {"tiny": TINY, "small": SMALL, "7b": W7B, "13b": W13B}

EPS = 1e-6
STD = 0.02                    # weights ~ N(0, 0.02), norm gains 1 + 0.1 N(0, 1)
N_SYS = 8                     # text tokens before the image (Eq. 3)


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _model_case(kind, model, dtype, layers, batch, vis, text, nodes, depth, topk, **more):
    return dict(kind=kind, model=model, dtype=dtype, layers=layers, batch=batch, vis=vis, text=text,
                nodes=nodes, depth=depth, topk=topk, **more)


def _linear_case(dtype, alloc, m, k, o, accumulate):
    return dict(kind="linear", dtype=dtype, alloc=alloc, m=m, k=k, o=o, accumulate=accumulate)


def listed():
    tree = dict(nodes=60, depth=6, topk=10)
    return [
        # the tiny reference model in fp32: the smallest calls, launches and latency
        dict(_model_case("draft_verify", "tiny", "f32", 2, 1, 64, 32, 16, 4, 4), name="tiny_f32_draft_verify"),
        # the tiny model in bf16, a whole short request of replayed steps
        dict(_model_case("generate", "tiny", "bf16", 2, 1, 64, 32, 16, 4, 4, steps=8, mode="tree", temperature=0.0),
             name="tiny_bf16_generate"),
        # fp32 at a generic small width: a prompt with an odd length, then sampled steps
        dict(_model_case("generate", "small", "f32", 4, 1, 256, 77, 24, 3, 6, steps=4, mode="sample", temperature=0.3),
             name="small_f32_sample"),
        # time to first token of one ordinary LLaVA prompt (576 visual + 64 text), 8 of the layers
        dict(_model_case("prefill", "7b", "bf16", 8, 1, 576, 64, **tree), name="prefill_7b"),
        # a ragged batch of prompts arriving together (batched serving), one and two images each
        dict(_model_case("prefill", "7b", "bf16", 2, 16, 1152, 512, **tree), name="prefill_7b_ragged16"),
        # the verify pass of the 60-node tree behind an ordinary prompt
        dict(_model_case("verify", "7b", "bf16", 8, 1, 576, 64, **tree), name="verify_7b"),
        # a chain draft's verify pass at the 13B width, odd prefix
        dict(_model_case("verify", "13b", "bf16", 4, 1, 576, 125, 7, 6, 1), name="verify_13b_chain"),
        # the verify pass behind a long multi-tile prefix (5 x 576 visual + 512 text)
        dict(_model_case("verify", "7b", "bf16", 4, 1, 2880, 512, **tree), name="verify_7b_long"),
        # the verify pass of batched serving: 16 ragged requests, 960 rows
        dict(_model_case("verify", "7b", "bf16", 2, 16, 1152, 512, **tree), name="verify_7b_batch16"),
        # a whole 7B request at full depth: prefill and 16 greedy tree steps
        dict(_model_case("generate", "7b", "bf16", 32, 1, 576, 64, steps=16, mode="tree", temperature=0.0, **tree),
             name="generate_7b"),
        # a projection of the caller's own weight: 576 visual rows into the model's width
        dict(_linear_case("bf16", True, 576, 4096, 4096, False), name="linear_projector"),
        # a few rows through a wide weight without an allocator, accumulating
        dict(_linear_case("bf16", False, 17, 4096, 11008, True), name="linear_noalloc_rows"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["draft_verify", "prefill", "prefill", "verify", "verify", "generate", "linear", "linear"])
    if kind == "linear":
        dtype, alloc = rng.choice([("bf16", True), ("bf16", True), ("bf16", False), ("bf16", False), ("f32", True)])
        big = dtype == "bf16"
        return _linear_case(dtype, alloc, _log_int(rng, 1, 1500 if big else 300),
                            8 * _log_int(rng, 8, 1376 if big else 256), _log_int(rng, 48, 22016 if big else 3000),
                            rng.random() < 0.5)
    if kind == "draft_verify":      # (fp32, or a chain: the frontier's order does not hang on rounding)
        if rng.random() < 0.5:
            return _model_case(kind, rng.choice(["tiny", "small"]), "f32", rng.randint(1, 3), rng.randint(1, 3),
                               _log_int(rng, 8, 300), _log_int(rng, 9, 100), rng.randint(5, 16), rng.randint(2, 4), 4)
        depth = rng.randint(2, 7)
        return _model_case(kind, rng.choice(["small", "7b"]), "bf16", rng.randint(1, 3), rng.randint(1, 4),
                           _log_int(rng, 16, 1152), _log_int(rng, 9, 512), depth + 1, depth, 1)
    f32 = rng.random() < 0.2
    model = rng.choice(["tiny", "small"]) if f32 else rng.choice(["small", "7b", "7b", "13b"])
    batch = rng.choice([1, 1, 1, 2, 5, 11])
    vis = rng.choice([0, _log_int(rng, 16, 700), 576, 576, 1152 if batch > 2 else 2880])
    text = _log_int(rng, 9, 512)
    nodes, depth, topk = rng.choice([(60, 6, 10), (rng.randint(17, 64), 5, 8), (rng.randint(65, 130), 6, 10),
                                     (rng.randint(2, 16), 4, 4), (1, 1, 1), (7, 6, 1)])
    layers = rng.randint(1, 2 if batch > 2 or f32 else 6)
    if f32:
        batch, vis, text = min(batch, 2), min(vis, 400), min(text, 128)
    more = {}
    if kind == "generate":
        batch = min(batch, 5)
        nodes = max(nodes, 2)
        depth = max(depth, 2) if topk > 1 else depth
        mode = rng.choice(["tree", "tree", "sample", "ar"])
        more = dict(steps=rng.randint(2, 8), mode=mode, temperature=0.3 if mode == "sample" else 0.0)
        nodes = min(nodes, topk + (depth - 1) * topk * topk + 1)
    return _model_case(kind, model, "f32" if f32 else "bf16", layers, batch, vis, text, nodes, depth, topk, **more)


def _lengths(c):
    """(visual, text) tokens of every request: ragged when there are several."""
    out = []
    for b in range(c["batch"]):
        if b == 0:
            out.append((c["vis"], c["text"]))
        else:
            lo = min(9, c["text"])
            out.append((c["vis"] if b % 2 else c["vis"] // 2, lo + (b * 167 + 29) % (c["text"] - lo + 1)))
    return out


def _max_seq(c):
    prompt = max(v + t for v, t in _lengths(c))
    return prompt + c.get("steps", 0) * (c["depth"] + 1) + c["nodes"] + 8


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _torch_dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _weights(c, seed):
    m, dt = MODELS[c["model"]], _torch_dtype(c)
    H, F, V = m["hidden"], m["ffn"], m["vocab"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 1)

    def mat(*shape):
        return torch.empty(shape, device="cuda", dtype=dt).normal_(0.0, STD, generator=g)

    def gain():
        return (1.0 + 0.1 * torch.randn(H, generator=g, device="cuda")).to(dt)

    def layer():
        w = {n: mat(H, H) for n in ("wq", "wk", "wv", "wo")}
        w["w_gate"], w["w_up"], w["w_down"] = mat(F, H), mat(F, H), mat(H, F)
        w["attn_norm"], w["mlp_norm"] = gain(), gain()
        return w

    return {"embed": mat(V, H), "lm_head": mat(V, H), "final_norm": gain(), "draft_fc": mat(H, 2 * H),
            "draft": layer(), "layers": [layer() for _ in range(c["layers"])]}


def _prompts(c, seed):
    """ids [B][stride] (-1 = visual slot), lengths, visual rows and their offsets."""
    m = MODELS[c["model"]]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 104729 + 2)
    lens = _lengths(c)
    stride = max(v + t for v, t in lens)
    text = torch.randint(0, m["vocab"], (c["batch"], stride), generator=g, device="cuda", dtype=torch.int32)
    offs, off = [], 0
    for b, (v, t) in enumerate(lens):
        p = min(N_SYS, t - 1)
        text[b, p:p + v] = -1
        offs.append(off)
        off += v
    vis = None
    if off:
        vis = (0.5 * torch.randn(off, m["hidden"], generator=g, device="cuda")).to(_torch_dtype(c))
    return text, [v + t for v, t in lens], vis, offs


def _planted(c, seed):
    """Tokens and parent links of one random tree per request (token 0 is the root's)."""
    r = random.Random(seed * 31 + 3)
    V, N, D = MODELS[c["model"]]["vocab"], c["nodes"], c["depth"]
    out = []
    for _ in range(c["batch"]):
        depth, parent = [0], [-1]
        for _i in range(1, N):
            p = r.choice([j for j in range(len(depth)) if depth[j] < D])
            parent.append(p)
            depth.append(depth[p] + 1)
        out.append(([r.randrange(V) for _i in range(N)], parent))
    return out


def _engine(c, w):
    m = MODELS[c["model"]]
    cfg = msd.msd_config(n_layers=c["layers"], hidden=m["hidden"], n_heads=m["heads"],
                         head_dim=m["hidden"] // m["heads"], ffn=m["ffn"], vocab=m["vocab"], rms_eps=EPS,
                         rope_base=10000.0, dtype=msd.MSD_BF16 if c["dtype"] == "bf16" else msd.MSD_F32,
                         max_batch=c["batch"], max_seq=_max_seq(c), tree_nodes=c["nodes"], tree_depth=c["depth"],
                         topk=c["topk"], draft_input=msd.DRAFT_INPUTS["embedding"])
    eng = msd.Engine(cfg, w)
    if c["dtype"] == "bf16":        # the context holds packed copies: the matrices may go
        eng.w = {"embed": w["embed"], "final_norm": w["final_norm"],
                 "norms": [(lw["attn_norm"], lw["mlp_norm"]) for lw in w["layers"] + [w["draft"]]]}
    return eng


def _plant(eng, c, seed):
    t = msd.Tree(c["batch"], c["nodes"])
    for b, (tokens, parent) in enumerate(_planted(c, seed)):
        eng.plant(t, b, tokens, parent)
    return t


def _linear_inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 15485863 + 4)
    dt = _torch_dtype(c)
    x = torch.randn(c["m"], c["k"], generator=g, device="cuda").to(dt)
    w = torch.empty(c["o"], c["k"], device="cuda", dtype=dt).normal_(0.0, STD, generator=g)
    y = torch.randn(c["m"], c["o"], generator=g, device="cuda")
    return x, w, y


def prepare(case, seed):
    c = dict(case)
    s = {"c": c}
    if c["kind"] == "linear":
        s["x"], s["w"], s["y"] = _linear_inputs(c, seed)
        if c["alloc"]:              # the handle that the call goes through
            h = _model_case("linear", "tiny", c["dtype"], 1, 1, 0, 9, 2, 1, 1)
            s["eng"] = _engine(h, _weights(h, seed))
        return s
    s["eng"] = eng = _engine(c, _weights(c, seed))
    s["ids"], s["lens"], s["vis"], s["offs"] = _prompts(c, seed)
    B, N, V = c["batch"], c["nodes"], MODELS[c["model"]]["vocab"]
    if c["kind"] != "prefill":
        s["logits"] = torch.zeros(B, N, V, device="cuda")
    if c["kind"] in ("verify", "generate"):
        s["tree"] = _plant(eng, c, seed)
    if c["kind"] in ("verify", "draft_verify"):
        root = eng.prefill(s["ids"], s["lens"], s["vis"], s["offs"])
        if c["kind"] == "verify":
            s["tree"].tokens.view(B, N)[:, 0].copy_(root)
    if c["kind"] == "draft_verify":
        D, k = c["depth"], c["topk"]
        s["record"] = {"logits": torch.zeros(B, D, k, V, device="cuda"),
                       "topk_ids": torch.zeros(B, D, k, k, dtype=torch.int32, device="cuda"),
                       "topk_logp": torch.zeros(B, D, k, k, device="cuda")}
    if c["kind"] == "generate" and c["mode"] == "sample":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed * 613 + 5)
        s["u"] = torch.rand(c["steps"], B, c["depth"] + 1, c["topk"] + 1, generator=g, device="cuda")
        s["u_step"] = torch.zeros_like(s["u"][0])
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _run_linear(s):
    c, x, w, y = s["c"], s["x"], s["w"], s["y"]
    if c["alloc"]:
        return s["eng"].linear(x, w, y, accumulate=c["accumulate"])
    st = msd.lib().msd_linear_noalloc(
        ctypes.c_void_p(x.data_ptr()), x.stride(0), c["m"], c["k"], ctypes.c_void_p(w.data_ptr()), c["o"],
        ctypes.c_void_p(y.data_ptr()), y.stride(0), int(c["accumulate"]),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if st != msd.MSD_OK:
        raise msd.MsdError(st, "msd_linear_noalloc", "")
    return y


def _cache(eng, name):
    """A context's cache as a tensor: a view of the context's own memory, so the
    tensor keeps the context."""
    view = eng.state()[name]
    view.engine = eng
    return view


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "linear":
        return _run_linear(s)
    eng = s["eng"]
    if c["kind"] == "draft_verify":
        t = eng.draft_tree(record=s["record"])
        argmax = eng.verify(logits=s["logits"])
        return {"tokens": t.tokens, "parent": t.parent, "depth": t.depth, "mask": t.mask, "argmax": argmax,
                "logits": s["logits"], **s["record"]}
    if c["kind"] == "verify":
        argmax = eng.verify(tree=s["tree"], logits=s["logits"])
        return {"argmax": argmax, "logits": s["logits"]}
    root = eng.prefill(s["ids"], s["lens"], s["vis"], s["offs"])
    if c["kind"] == "prefill":
        return {"root": root, "target_kv": _cache(eng, "target_kv"), "draft_kv": _cache(eng, "draft_kv")}
    emitted = [root.clone()]
    for i in range(c["steps"]):
        if c["mode"] == "ar":
            emitted.append(eng.ar_step().clone())
            continue
        if c["mode"] == "sample":
            s["u_step"].copy_(s["u"][i])
            path, n, bonus = eng.step_sample(c["temperature"], s["u_step"])
        else:
            path, n, bonus = eng.step()
        emitted += [torch.cat((path, n, bonus))]
    B, N = c["batch"], c["nodes"]
    s["tree"].tokens.view(B, N)[:, 0].copy_(emitted[-1][-B:])
    argmax = eng.verify(tree=s["tree"], logits=s["logits"])
    return {"emitted": torch.cat(emitted), "argmax": argmax, "logits": s["logits"],
            "target_kv": _cache(eng, "target_kv")}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _esz(c):
    return 2 if c["dtype"] == "bf16" else 4


def _layer_params(m):
    return 4 * m["hidden"] ** 2 + 3 * m["hidden"] * m["ffn"]


def _pass_work(c, layers, rows, head_rows, keys, extra_params=0):
    """Weights once, the K/V each request sees (summed: keys) read once per layer,
    the rows' own K/V written, head_rows rows of logits."""
    m, e = MODELS[c["model"]], _esz(c)
    H, V = m["hidden"], m["vocab"]
    params = layers * _layer_params(m) + extra_params
    head = H * V if head_rows else 0
    b = e * (params + head) + e * layers * 2 * H * (keys + rows) + rows * H * e + 4 * head_rows * V
    f = 2.0 * rows * params + 2.0 * head_rows * head
    return b, f


def _attn_flops(c, layers, pairs):
    return 4.0 * layers * pairs * MODELS[c["model"]]["hidden"]


def _prefill_work(c):
    H = MODELS[c["model"]]["hidden"]
    L = [v + t for v, t in _lengths(c)]
    rows, pairs = sum(L), sum(x * (x + 1) / 2.0 for x in L)
    b, f = _pass_work(c, c["layers"], rows, c["batch"], 0)
    b2, f2 = _pass_work(c, 1, rows - c["batch"], 0, 0, 2 * H * H)
    return b + b2, f + f2 + _attn_flops(c, c["layers"] + 1, pairs)


def _verify_work(c, grown=0, nodes=None):
    N, L = c["nodes"] if nodes is None else nodes, [v + t + grown for v, t in _lengths(c)]
    b, f = _pass_work(c, c["layers"], c["batch"] * N, c["batch"] * N, sum(L))
    return b, f + _attn_flops(c, c["layers"], sum(N * (x + N / 2.0) for x in L))


def _draft_work(c, grown=0):
    H, k = MODELS[c["model"]]["hidden"], c["topk"]
    L = [v + t + grown for v, t in _lengths(c)]
    b = f = 0.0
    for p in range(c["depth"]):
        rows = c["batch"] * (1 if p == 0 else k)
        b1, f1 = _pass_work(c, 1, rows, rows, sum(L), 2 * H * H)
        b, f = b + b1, f + f1 + _attn_flops(c, 1, rows / c["batch"] * sum(L))
    return b, f


def work(case):
    c = case
    if c["kind"] == "linear":
        e = _esz(c)
        b = e * (c["m"] * c["k"] + c["o"] * c["k"]) + 4 * c["m"] * c["o"] * (2 if c["accumulate"] else 1)
        return {"bytes": b, "flops": 2.0 * c["m"] * c["k"] * c["o"]}
    if c["kind"] == "prefill":
        b, f = _prefill_work(c)
    elif c["kind"] == "verify":
        b, f = _verify_work(c)
    elif c["kind"] == "draft_verify":
        b, f = (x + y for x, y in zip(_draft_work(c), _verify_work(c)))
    else:
        b, f = _prefill_work(c)
        for i in range(c["steps"]):
            parts = [_verify_work(c, i, 1 if c["mode"] == "ar" else None)]
            if c["mode"] != "ar":
                parts.append(_draft_work(c, i))
            b, f = b + sum(x for x, _ in parts), f + sum(x for _, x in parts)
        b1, f1 = _verify_work(c, c["steps"])
        b, f = b + b1, f + f1
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    c = case
    if c["kind"] == "linear":                   # exact bf16 (or fp32) products, fp32 sums
        return {"rel": 4e-6, "max": 1e-4}
    if c["kind"] == "prefill":                  # the caches' bf16 values: a sum that rounds the other way moves one by 2^-8
        return {"rel": 4e-3, "max": 2e-2, "differ": 0.0} if c["dtype"] == "bf16" else {"rel": 2e-5, "max": 1e-3, "differ": 0.0}
    # logits of fp32 layers, or of split-bf16 ones (about 2^-17 a value, through every layer); tokens may tie
    t = {"rel": 3e-4, "max": 3e-3, "differ": 0.01} if c["dtype"] == "bf16" else {"rel": 2e-5, "max": 2e-4, "differ": 0.01}
    if c["kind"] == "generate" and c["dtype"] == "bf16":
        t.update(rel=4e-3, max=2e-2)            # the returned cache's bf16 values, as above
    if c["kind"] == "draft_verify":             # the draft feeds on its own un-normalised feature
        t.update(rel=1e-3 if c["dtype"] == "bf16" else 1e-4, max=1e-2 if c["dtype"] == "bf16" else 1e-3)
    return t


# ---------------------------------------------------------------------------
# The same values in 64 bits
# ---------------------------------------------------------------------------
def _rms(x, g):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + EPS) * g.double()


def _rope(x, pos):
    """x [R][heads][hd], rotate-half pairs (i, i + hd/2)."""
    half = x.shape[-1] // 2
    th = 10000.0 ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    a = pos.double()[:, None] * th
    cos, sin = torch.cos(a)[:, None], torch.sin(a)[:, None]
    x0, x1 = x[..., :half], x[..., half:]
    return torch.cat((x0 * cos - x1 * sin, x1 * cos + x0 * sin), -1)


def _decoder_layer(lw, x, heads, pos, seen, K0=None, V0=None):
    """One pre-norm layer over rows x: every row sees the whole cache (K0, V0)
    and the rows of this block that `seen` allows. Returns x, K, V of the rows."""
    R, H = x.shape
    hd = H // heads
    n = _rms(x, lw["attn_norm"])
    q, k, v = ((n @ lw[w].double().T).view(R, heads, hd) for w in ("wq", "wk", "wv"))
    q, k = _rope(q, pos), _rope(k, pos)
    ka, va = (k, v) if K0 is None else (torch.cat((K0, k)), torch.cat((V0, v)))
    out = torch.empty_like(q)
    for h in range(heads):
        s = q[:, h] @ ka[:, h].T / math.sqrt(hd)
        s[:, s.shape[1] - R:].masked_fill_(~seen, -math.inf)
        out[:, h] = torch.softmax(s, -1) @ va[:, h]
    x = x + out.reshape(R, H) @ lw["wo"].double().T
    n = _rms(x, lw["mlp_norm"])
    a = torch.nn.functional.silu(n @ lw["w_gate"].double().T) * (n @ lw["w_up"].double().T)
    return x + a @ lw["w_down"].double().T, k, v


def _target_prefill(c, w, ids, vis):
    heads = MODELS[c["model"]]["heads"]
    is_vis = ids < 0
    emb = w["embed"].double()[ids.clamp(min=0).long()]
    if is_vis.any():
        emb[is_vis] = vis.double()
    L = ids.shape[0]
    pos = torch.arange(L, device=ids.device)
    seen = torch.ones(L, L, dtype=torch.bool, device=ids.device).tril()
    x, kv = emb, []
    for lw in w["layers"]:
        x, k, v = _decoder_layer(lw, x, heads, pos, seen)
        kv.append((k, v))
    return _rms(x, w["final_norm"]), kv, emb, is_vis, pos, seen


def _store(dst, b, k, v):
    """K and V of a request's first positions into [2][B][heads][max_seq][hd]."""
    dst[0, b, :, :k.shape[0]] = k.transpose(0, 1)
    dst[1, b, :, :v.shape[0]] = v.transpose(0, 1)


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "linear":
        x, w, y = _linear_inputs(c, seed)
        r = x.double() @ w.double().T
        return r + y.double() if c["accumulate"] else r
    rows = sum(v + t for v, t in _lengths(c))
    flops = 2.0 * rows * _layer_params(MODELS[c["model"]]) * (c["layers"] + 1)
    if c["kind"] in ("draft_verify", "generate") or flops > 4e12:
        return None     # (trees and tokens of the fp32 and whole-request cases have no such value)
    m, B, N = MODELS[c["model"]], c["batch"], c["nodes"]
    heads, hd = m["heads"], m["hidden"] // m["heads"]
    w = _weights(c, seed)
    ids, lens, vis, offs = _prompts(c, seed)
    out = {}
    if c["kind"] == "prefill":
        S = _max_seq(c)
        tkv = torch.zeros(c["layers"], 2, B, heads, S, hd, dtype=torch.float64, device="cuda")
        dkv = torch.zeros(2, B, heads, S, hd, dtype=torch.float64, device="cuda")
    else:
        logits = torch.zeros(B, N, m["vocab"], dtype=torch.float64, device="cuda")
        planted = _planted(c, seed)
    for b in range(B):
        L = lens[b]
        n_vis = _lengths(c)[b][0]
        h, kv, emb, is_vis, pos, seen = _target_prefill(
            c, w, ids[b, :L], None if vis is None else vis[offs[b]:offs[b] + n_vis])
        if c["kind"] == "prefill":
            for layer, (k, v) in enumerate(kv):
                _store(tkv[layer], b, k, v)
            if L > 1:           # draft rows 0 .. L-2: f_down(Concat(h, e_next)) at text, e at visual positions
                f = torch.cat((h[:-1], emb[1:]), -1) @ w["draft_fc"].double().T
                f = torch.where(is_vis[:-1, None], emb[:-1], f)
                _, k, v = _decoder_layer(w["draft"], f, heads, pos[:-1], seen[:-1, :-1])
                _store(dkv, b, k, v)
            continue
        tokens, parent = planted[b]
        root = int(torch.argmax(h[-1] @ w["lm_head"].double().T))
        depth, mask = [0], torch.eye(N, dtype=torch.bool, device="cuda")
        for i in range(1, N):
            depth.append(depth[parent[i]] + 1)
            mask[i] |= mask[parent[i]]
        x = w["embed"].double()[torch.tensor([root] + tokens[1:], device="cuda")]
        tpos = L + torch.tensor(depth, device="cuda")
        for lw, (k, v) in zip(w["layers"], kv):
            x, _, _ = _decoder_layer(lw, x, heads, tpos, mask, k, v)
        logits[b] = _rms(x, w["final_norm"]) @ w["lm_head"].double().T
    if c["kind"] == "prefill":
        return {"root": None, "target_kv": tkv, "draft_kv": dkv}
    return {"argmax": None, "logits": logits}
