"""Workloads the library is measured on: what a program that serves or studies a long-context model
asks of it, through the public binding.

Kinds of case (``"kind"``):
  layer    mixkv_compress_layer: one layer's cache compressed as soon as its prefill is done
  layers   mixkv_compress_layers[_budgeted]: the caches of all layers at the end of prefill
  scores   mixkv_scores, then mixkv_select on what it returned: the two-step interface of a program
           that looks at (or edits) the scores before it selects
  decode   mixkv_decode_attention: one new token over the compact cache
  sim      mixkv_similarity_map: the redundancy heat map of the keys of a layer

Lengths of a ragged batch are written as text ("4096" or "5003,1291"), so that a case is a dict of
plain values.  Keys follow the statistics of ``paper_2510_20707_b200.synth`` (its calibrated variant)
and are drawn on the GPU.
"""
import math
import random

import torch

from paper_2510_20707_b200 import binding

D = 128
VISION_X = (0.4, 1.2, 2.4, 10.0)   # squared norm of a head's shared key offset, in units of d


def listed():
    base = dict(H=4, G=7, W=32, pool=7, pool_mode=0, vnorm=1, mode="fixed", data="image")
    return [
        # the smallest prefill: one image and a question, one layer per call (launches and host time)
        dict(base, name="layer_small", kind="layer", layers=1, lens="1024", B=64),
        # a long video, one call per layer as the layers finish
        dict(base, name="layer_video", kind="layer", layers=1, lens="32768", B=256, data="video"),
        # an ordinary image prompt, all 28 layers at the end of prefill
        dict(base, name="layers_image", kind="layers", layers=28, lens="4096", B=128),
        # the long video, all layers at once: the largest call, the benchmark's default workload
        dict(base, name="layers_video", kind="layers", layers=28, lens="32768", B=256, data="video"),
        # a served batch of eight ragged prompts with head-adaptive budgets
        dict(base, name="layers_batch", kind="layers", layers=28, mode="adaptive", B=128,
             lens="5639,5104,2112,2908,7334,2865,5376,2051"),
        # a text-only model with eight KV heads and four query heads each
        dict(base, name="layers_text", kind="layers", layers=32, H=8, G=4, lens="16384", B=256,
             data="text"),
        # budgets that fall with depth (PyramidKV manner), three prompts of odd lengths
        dict(base, name="layers_schedule", kind="layers", layers=28, mode="schedule", B=256,
             lens="3001,1777,6143"),
        # scores handed to the caller, then its selection; max pooling and the key-norm variant
        dict(base, name="scores_select", kind="scores", layers=1, H=8, G=4, mode="adaptive", B=160,
             lens="5003,1291,12007", pool_mode=1, vnorm=2),
        # a decode step as a model runs it: one layer, one sequence
        dict(name="decode_layer", kind="decode", layers=1, batch=1, H=4, G=7, B=512, ragged=False),
        # a decode step of a served batch over ragged (adaptive) caches, all layers
        dict(name="decode_batch", kind="decode", layers=28, batch=8, H=4, G=7, B=512, ragged=True),
        # the heat map of a long video's keys at 16 tokens per cell
        dict(name="sim_fine", kind="sim", H=4, L=32768, block=16),
        # the same at a resolution that can be looked at: a cell per quarter of a frame
        dict(name="sim_coarse", kind="sim", H=4, L=32768, block=256),
    ]


# -------------------------------------------------------------------------------------- drawn cases
MOST_TOKENS = 28 * 4 * 32768       # (layer, head, token) triples of the largest listed call
GW = ((7, 32), (7, 32), (4, 32), (4, 32), (8, 16), (2, 32), (1, 32), (5, 32), (6, 32), (7, 16), (15, 16),
      (3, 64), (1, 16))


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_compress(rng, kind):
    G, W = rng.choice(GW)
    H = rng.choice((1, 2, 4, 4, 8))
    layers = 1 if kind != "layers" else _log_int(rng, 2, 40)
    batch = 1 if rng.random() < 0.5 else rng.randint(2, 8)
    most = min(49152, MOST_TOKENS // (layers * H * batch))
    top = _log_int(rng, 600, most)
    lens = [top] + [rng.randint(max(400, top // 4), top) for _ in range(batch - 1)]
    short = min(lens)
    mode = rng.choice(("fixed", "fixed", "adaptive", "schedule" if kind == "layers" else "fixed"))
    # a twentieth to a quarter of the shortest prompt, within the budgets in use
    room = short // 4 if mode != "adaptive" else short // (2 * H)
    B = max(W + 16, min(1024, _log_int(rng, 40, max(41, room))))
    return dict(kind=kind, layers=layers, H=H, G=G, W=W, lens=",".join(str(x) for x in lens), B=B,
                mode=mode, pool=rng.choice((7, 7, 7, 5, 1)), pool_mode=int(rng.random() < 0.2),
                vnorm=rng.choice((1, 1, 1, 0, 2)), data=rng.choice(("image", "video", "text")))


def _draw_decode(rng):
    H = rng.choice((1, 2, 4, 8))
    layers = rng.choice((1, 1, 28, 32, rng.randint(2, 40)))
    batch = rng.choice((1, 1, rng.randint(2, 16)))
    most = min(8192, (1 << 21) // (layers * batch * H))
    return dict(kind="decode", layers=layers, batch=batch, H=H, G=rng.choice((1, 4, 7, 7, 8, 12, 16)),
                B=_log_int(rng, 64, most), ragged=rng.random() < 0.5)


def _draw_sim(rng):
    H = rng.choice((1, 2, 4, 8))
    block = rng.choice((1, 2, 4, 8, 16, 16, _log_int(rng, 17, 1024), _log_int(rng, 17, 1024)))
    most = min(40000, 8192 * block if H <= 4 else 5792 * block, int(32768 * math.sqrt(4 / H)))
    return dict(kind="sim", H=H, L=_log_int(rng, 512, most), block=block)


def draw(rng: random.Random):
    kind = rng.choice(("layer", "layer", "layers", "layers", "layers", "layers", "scores", "decode",
                       "decode", "sim", "sim"))
    if kind == "decode":
        return _draw_decode(rng)
    if kind == "sim":
        return _draw_sim(rng)
    return _draw_compress(rng, kind)


# ------------------------------------------------------------------------------------------- inputs
def _lens(case):
    return [int(x) for x in case["lens"].split(",")]


def _params(case):
    adaptive = case["mode"] == "adaptive"
    return binding.Params(kv_heads=case["H"], gqa_ratio=case["G"], window=case["W"],
                          pool_kernel=case["pool"], pool_mode=case["pool_mode"],
                          use_vnorm=case["vnorm"], budget=case["B"], budget_mode=int(adaptive))


def _randn(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda")


def _offsets(gen, H, data):
    """The offset that all keys of a head share [H, d]: it sets the head's mean pairwise cosine
    (0.2 .. 0.4 for text, 0.26 .. 0.9 for vision)."""
    m = _randn(gen, H, D)
    if data == "text":
        rho = [0.2 + 0.2 * h / max(H - 1, 1) for h in range(H)]
        x = [r / (1 - r) for r in rho]
    else:
        x = [VISION_X[h % len(VISION_X)] for h in range(H)]
    x = torch.tensor(x, device="cuda").unsqueeze(1) * D
    return m * (x.sqrt() / m.norm(dim=1, keepdim=True))


def _keys(gen, H, L, data):
    """Keys [H, L, d] of one sequence: vision tokens scatter around centroids (of the image, or of
    each of 32 frames with slow drift between them), the last eighth is text."""
    K = _randn(gen, H, L, D)
    if data != "text":
        frames, cent = (32, 32) if data == "video" else (1, 64)
        nv = L - L // 8
        c = _randn(gen, frames, H, cent, D)
        for f in range(1, frames):
            c[f].mul_(math.sqrt(1 - 0.98 ** 2)).add_(c[f - 1], alpha=0.98)
        frame = torch.arange(nv, device="cuda") * frames // nv
        pick = torch.randint(0, cent, (H, nv), generator=gen, device="cuda")
        head = torch.arange(H, device="cuda").unsqueeze(1)
        K[:, :nv].mul_(0.35).add_(c[frame.unsqueeze(0), head, pick])
    return K.add_(_offsets(gen, H, data).unsqueeze(1))


def _prepare_compress(case, gen):
    p, lens, NL = _params(case), _lens(case), case["layers"]
    H, batch, total = case["H"], len(lens), sum(lens)
    cu = [0]
    for n in lens:
        cu.append(cu[-1] + n)
    bf16 = dict(dtype=torch.bfloat16, device="cuda")
    i32 = dict(dtype=torch.int32, device="cuda")
    K = torch.empty((NL, H, total, D), **bf16)
    for l in range(NL):
        for b, n in enumerate(lens):
            K[l, :, cu[b]:cu[b + 1]] = _keys(gen, H, n, case["data"])
    V = torch.empty_like(K).normal_(generator=gen)
    Q = torch.empty((NL, batch, H * case["G"], case["W"], D), **bf16).normal_(generator=gen)
    state = {"kind": case["kind"], "p": p, "cu": cu if batch > 1 else None, "budgets": None}
    if case["mode"] == "schedule":
        rows = binding.layer_budget_schedule(NL, case["B"], case["W"], 500)
        p.budget = rows[0]
        state["budgets"] = torch.tensor(rows, **i32).unsqueeze(1).repeat(1, batch * H).contiguous()
    # a server keeps the workspace and the output buffers from call to call
    nbytes = binding.workspace_size_layers(p, NL, batch, total, max(lens))
    state["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    if case["kind"] == "scores":
        state.update(K=K[0], V=V[0], Q=Q[0])
        return state
    rows = batch * H * p.budget
    out = {"K_out": torch.zeros((NL, rows, D), **bf16), "V_out": torch.zeros((NL, rows, D), **bf16),
           "out_row_offsets": torch.zeros((NL, batch * H + 1), **i32), "status": torch.zeros(1, **i32)}
    if case["kind"] == "layer":
        K, V, Q = K[0], V[0], Q[0]
        out = {k: v if k == "status" else v[0] for k, v in out.items()}
    state.update(K=K, V=V, Q=Q, out=out)
    # the kept rows are copies of input rows, bit for bit: looked at as whole numbers
    state["result"] = {"K_out": out["K_out"].view(torch.int16), "V_out": out["V_out"].view(torch.int16),
                       "out_row_offsets": out["out_row_offsets"], "status": out["status"]}
    return state


def _prepare_decode(case, gen, seed):
    NL, batch, H, B = case["layers"], case["batch"], case["H"], case["B"]
    rows = batch * H * B
    bf16 = dict(dtype=torch.bfloat16, device="cuda")
    K = torch.empty((NL, rows, D), **bf16).normal_(generator=gen)
    V = torch.empty((NL, rows, D), **bf16).normal_(generator=gen)
    q = torch.empty((NL, batch, H * case["G"], D), **bf16).normal_(generator=gen)
    # rows of every (layer, sequence, head): B each, or B * H per sequence shared unevenly with a
    # fifth of B for every head, as head-adaptive budgets leave them
    counts = torch.full((NL, batch, H), B, dtype=torch.int64)
    if case["ragged"] and H > 1:
        floor, free = B // 5, H * (B - B // 5)
        cut = torch.rand((NL, batch, H - 1), generator=torch.Generator().manual_seed(seed))
        cut = (cut * (free + 1)).long().clamp(max=free).sort(dim=2).values
        ends = torch.cat([torch.zeros(NL, batch, 1, dtype=torch.int64), cut,
                          torch.full((NL, batch, 1), free, dtype=torch.int64)], dim=2)
        counts = floor + ends.diff(dim=2)
    offs = torch.cat([torch.zeros(NL, 1, dtype=torch.int64), counts.reshape(NL, -1).cumsum(1)], dim=1)
    return {"kind": "decode", "K": K, "V": V, "q": q, "offs": offs.int().cuda(), "H": H, "G": case["G"],
            "max_rows": int(counts.max())}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "decode":
        return _prepare_decode(case, gen, seed)
    if case["kind"] == "sim":
        X = _keys(gen, case["H"], case["L"], "video").bfloat16()
        return {"kind": "sim", "X": X, "block": case["block"]}
    return _prepare_compress(case, gen)


# ---------------------------------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "decode":
        return binding.decode_attention(state["K"], state["V"], state["offs"], state["q"], state["H"],
                                        state["G"], state["max_rows"])
    if kind == "sim":
        return binding.similarity_map(state["X"], state["block"])
    if kind == "layer":
        binding.compress_layer(state["K"], state["V"], state["Q"], state["p"], cu_seqlens=state["cu"],
                               workspace=state["ws"], out=state["out"], want_aux=False)
        return state["result"]
    if kind == "layers":
        binding.compress_layers(state["K"], state["V"], state["Q"], state["p"], cu_seqlens=state["cu"],
                                workspace=state["ws"], out=state["out"], want_aux=False,
                                head_budgets=state["budgets"])
        return state["result"]
    s = binding.scores(state["K"], state["V"], state["Q"], state["p"], cu_seqlens=state["cu"],
                       workspace=state["ws"])
    sel = binding.select(s["s_comp"], state["p"], cu_seqlens=state["cu"], workspace=state["ws"])
    return {"scores": s, "select": sel}


def work(case):
    if case["kind"] == "decode":
        units = case["layers"] * case["batch"] * case["H"]
        rows = units * case["B"]
        return {"bytes": rows * 2 * D * 2 + units * case["G"] * D * (2 + 4) + 4 * units,
                "flops": 4.0 * rows * case["G"] * D}
    if case["kind"] == "sim":
        H, L, T = case["H"], case["L"], -(-case["L"] // case["block"])
        # the map is symmetric, and a cell is the product of two sums of unit rows
        return {"bytes": H * (L * D * 2 + T * T * 4), "flops": float(H) * (T * (T + 1) * D + 5 * L * D)}
    H, W, NQ, lens = case["H"], case["W"], case["G"] * case["W"], _lens(case)
    B, NL = case["B"], case["layers"]
    kv = 2 if case["vnorm"] == 1 else 1
    nbytes = sum(H * (kv * L * D * 2 + NQ * D * 2) for L in lens)
    kept = sum(H * min(B - W, L - W) for L in lens)
    if case["kind"] == "scores":
        nbytes += sum(3 * H * (L - W) * 4 for L in lens) + kept * 4 + sum(H * (L - W) * 4 for L in lens)
    else:
        # rows gathered: read and written (without value norms, V is read here for the first time)
        nbytes += (kept + len(lens) * H * W) * 2 * 2 * D * 2
    flops = sum(H * (2.0 * L * NQ * D + kv * 2.0 * L * D + 4.0 * L * D) for L in lens)
    return {"bytes": NL * nbytes, "flops": NL * flops}


def tolerance(case):
    # fp32 sums and exponentials throughout; a kept row may change where two scores tie to fp32 rounding
    if case["kind"] in ("decode", "sim"):
        return {"rel": 1e-5}
    return {"rel": 1e-5, "differ": 0.01}
