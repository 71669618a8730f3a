"""Performance cases of the packed-encoder hot path: what one encoder microbatch costs through the public entry points.

Three kinds of pass, told apart by ``case["kind"]``:

  step     ``hotpath.run_step``: segment plan and its upload, attention forward, attention backward (trained encoder) and
           the merge of the encoder rows into the LLM input, one microbatch.  The plan is part of the pass because every
           microbatch brings its own patch counts.
  encoder  ``seg_plan`` + ``encoder_fwd`` over a stack of layers and, for a trained encoder, the zeroing of the flat
           gradient bucket and ``encoder_bwd``: one training step of the region with one microbatch.
  seam     ``merge_tokens`` + ``merge_tokens_bwd``: both directions of the local Replicated -> Sharded seam.

A case holds plain values only.  Patch counts come from the repository's own workload recipes (tiny, vit_l, qwen2vl, video,
mix) or from ``packed``: ``images`` segments with log-uniform patch counts in ``[lo, hi]``; ``structure`` seeds them, so
that the sizes of a case never depend on the seed of its values.
"""
import math
import random

import torch

from paper_2607_03229_b200 import binding as B
from paper_2607_03229_b200 import dist as D
from paper_2607_03229_b200 import hotpath as H
from paper_2607_03229_b200 import workloads as W

LN_EPS = 1e-6


def listed():
    return [
        # One small microbatch (four icons, 229 tokens): launches, the host plan and marshalling are all there is to pay.
        {"name": "step_tiny", "kind": "step", "recipe": "tiny", "structure": 1, "trained": True},
        # A text-heavy batch: 10 % image tokens in eight 8192-token sequences, trained, merged at the LLM's hidden size.
        {"name": "step_mix10", "kind": "step", "recipe": "mix", "fraction": 0.10, "seqs": 8, "seq_len": 8192,
         "llm_hidden": 4096, "structure": 5, "trained": True},
        # Thumbnails: 200 images of 64-256 patches at head_dim 80, trained; no segment fills more than two tiles.
        {"name": "step_thumbs", "kind": "step", "recipe": "video", "small": 200, "clips": 0, "structure": 4, "trained": True},
        # The ordinary training microbatch: 32 images of 224-896 pixels, 16 heads of 64, trained, merged into the LLM input.
        {"name": "step_vit_l", "kind": "step", "recipe": "vit_l", "images": 32, "llm_tokens": 131072, "structure": 2,
         "trained": True},
        # A frozen encoder on long-tailed native resolutions, 16 heads of 80: the forward alone.
        {"name": "step_qwen2vl_frozen", "kind": "step", "recipe": "qwen2vl", "total": 65536, "structure": 3, "trained": False},
        # The largest microbatch: 200 small images and four 16384-patch clips, head_dim 80, trained.
        {"name": "step_video_tail", "kind": "step", "recipe": "video", "small": 200, "clips": 4, "structure": 4, "trained": True},
        # One image of odd size through a frozen 24-layer encoder: serving latency, every product smaller than the chip.
        {"name": "encoder_one_image", "kind": "encoder", "recipe": "packed", "images": 1, "lo": 777, "hi": 777, "structure": 7,
         "heads": 16, "head_dim": 64, "layers": 24, "rope": False, "trained": False},
        # A small training microbatch (five ragged images, a few thousand tokens) through four layers, forward and backward.
        {"name": "encoder_small_trained", "kind": "encoder", "recipe": "packed", "images": 5, "lo": 300, "hi": 1500,
         "structure": 8, "heads": 16, "head_dim": 64, "layers": 4, "rope": False, "trained": True},
        # One layer of a frozen encoder over the ordinary microbatch: the projections at full size.
        {"name": "encoder_vit_l_frozen", "kind": "encoder", "recipe": "vit_l", "images": 32, "structure": 2, "heads": 16,
         "head_dim": 64, "layers": 1, "rope": False, "trained": False},
        # The same layer trained: input, weight, bias and norm gradients.
        {"name": "encoder_vit_l_trained", "kind": "encoder", "recipe": "vit_l", "images": 32, "structure": 2, "heads": 16,
         "head_dim": 64, "layers": 1, "rope": False, "trained": True},
        # A trained layer with rotary encoding at head_dim 80 (hidden 1280) over 65536 tokens of long-tailed images.
        {"name": "encoder_qwen2vl_trained", "kind": "encoder", "recipe": "qwen2vl", "total": 65536, "structure": 3, "heads": 16,
         "head_dim": 80, "layers": 1, "rope": True, "trained": True},
        # The seam alone at its largest: 75 % image tokens, rows of 4096, gathered forward and scattered back.
        {"name": "seam_mix75", "kind": "seam", "recipe": "mix", "fraction": 0.75, "seqs": 8, "seq_len": 8192,
         "llm_hidden": 4096, "structure": 5, "trained": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        structure = rng.randrange(1 << 20)
        trained = rng.random() < 0.6
        kind = rng.choice(["step"] * 4 + ["encoder"] * 5 + ["seam"])
        mix = {"recipe": "mix", "fraction": round(rng.uniform(0.05, 0.75), 3), "seqs": rng.randint(1, 8),
               "seq_len": 8 * _log_int(rng, 128, 1024), "llm_hidden": rng.choice([1024, 2048, 4096]), "structure": structure}
        lo = _log_int(rng, 16, 4096)
        packed = {"recipe": "packed", "images": _log_int(rng, 1, 256), "lo": lo, "hi": min(16384, _log_int(rng, lo, 16 * lo)),
                  "structure": structure, "heads": rng.choice([4, 8, 16]), "head_dim": rng.choice([64, 80])}
        if kind == "seam":
            case = dict(mix, kind="seam", trained=True)
        elif kind == "encoder":
            case = dict(packed, kind="encoder", layers=_log_int(rng, 1, 24), rope=rng.random() < 0.5, trained=trained)
        elif rng.random() < 0.4:
            case = dict(mix, kind="step", trained=trained)
        else:
            case = dict(packed, kind="step", trained=trained)
        w = _workload(case)
        tokens = w.total_tokens * case.get("layers", 1)
        if 0 < tokens <= 65536 and work(case)["flops"] <= 1.2e13:
            return case


def _workload(case):
    """Patch counts, heads and merge positions of a case as one of the repository's workloads."""
    recipe, seed = case["recipe"], W.BASE_SEED + case["structure"]
    if recipe == "tiny":
        return W.tiny(seed)
    if recipe == "vit_l":
        return W.vit_l(seed, case["images"], case.get("llm_tokens", 131072))
    if recipe == "qwen2vl":
        return W.qwen2vl(seed, case["trained"], case["total"])
    if recipe == "video":
        w = W.video_tail(seed, case["small"], case["clips"])
        w.trained = case["trained"]
        return w
    if recipe == "mix":
        return W.modality_mix(case["fraction"], seed, case["trained"], case["seqs"], case["seq_len"], case["llm_hidden"])
    rng = random.Random(case["structure"])
    counts = [_log_int(rng, case["lo"], case["hi"]) for _ in range(case["images"])]
    return W.Workload("packed", seed, counts, case["heads"], case["head_dim"], case["trained"])


def _normal(gen, shape, std=1.0, mean=0.0):
    return (torch.randn(shape, device="cuda", generator=gen) * std + mean).to(torch.bfloat16)


def _prepare_step(w, gen):
    shape = (w.total_tokens, w.n_heads, w.head_dim)
    emb = src = None
    if w.merge_hidden is not None:
        emb = _normal(gen, (w.n_llm_tokens, w.merge_hidden))
        if w.merge_hidden != w.n_heads * w.head_dim:
            src = _normal(gen, (w.total_tokens, w.merge_hidden))    # stands for the projector's output
    q, k, v = (_normal(gen, shape) for _ in range(3))
    dout = _normal(gen, shape) if w.trained else None
    return {"kind": "step", "w": w, "buf": H.allocate(w, "cuda", q=q, k=k, v=v, dout=dout, llm_embeds=emb, merge_src=src)}


def _prepare_seam(w, gen):
    rows, width = w.total_tokens, w.merge_hidden
    return {"kind": "seam", "enc": _normal(gen, (rows, width)), "emb": _normal(gen, (w.n_llm_tokens, width)),
            "d_emb": _normal(gen, (w.n_llm_tokens, width)), "d_enc": torch.empty((rows, width), dtype=torch.bfloat16, device="cuda"),
            "pos": torch.from_numpy(w.positions).cuda(), "status": torch.zeros(4, dtype=torch.int32, device="cuda")}


def _prepare_encoder(case, w, gen):
    heads, n_layers, trained = case["heads"], case["layers"], case["trained"]
    hidden = heads * case["head_dim"]
    ffn, T = 4 * hidden, w.total_tokens
    mode = B.TRAINED if trained else B.FROZEN
    layers = []
    for _ in range(n_layers):
        params = {}
        for name, shape in D.LAYER_PARAM_SHAPES:
            shp = shape(hidden, ffn)
            if name.startswith("w_"):
                params[name] = _normal(gen, shp, shp[1] ** -0.5)
            else:
                params[name] = _normal(gen, shp, 0.1, 1.0 if name.endswith("gamma") else 0.0)
        layers.append(B.LayerWeights.from_tensors(**params))
    x = _normal(gen, (T, hidden))
    state = {"kind": "encoder", "w": w, "mode": mode, "heads": heads, "ffn": ffn, "layers": layers, "x": x, "y": torch.empty_like(x),
             "ws": torch.empty(B.encoder_workspace_bytes(n_layers, T, hidden, ffn, mode), dtype=torch.uint8, device="cuda"),
             "status": torch.zeros(4, dtype=torch.int32, device="cuda"), "lse": None, "rope": None}
    if case["rope"]:
        state["rope"] = tuple(torch.from_numpy(t).cuda() for t in W.rope2d_tables(w.patch_counts, case["head_dim"]))
    if trained:
        bucket, views = D.alloc_grad_bucket(n_layers, hidden, ffn)
        state.update(lse=torch.empty((n_layers, heads, T), dtype=torch.float32, device="cuda"), dy=_normal(gen, (T, hidden)),
                     dx=torch.empty_like(x), bucket=bucket, grads=[B.LayerGrads.from_tensors(**v) for v in views],
                     ws_bwd=torch.empty(B.encoder_bwd_workspace_bytes(T, hidden, heads, ffn), dtype=torch.uint8, device="cuda"))
    return state


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    w = _workload(case)
    if case["kind"] == "step":
        return _prepare_step(w, gen)
    if case["kind"] == "seam":
        return _prepare_seam(w, gen)
    return _prepare_encoder(case, w, gen)


def run(s):
    if s["kind"] == "step":
        buf = s["buf"]
        H.run_step(s["w"], buf)
        return [buf.o, buf.lse, buf.dq, buf.dk, buf.dv, buf.llm_embeds]
    if s["kind"] == "seam":
        B.merge_tokens(s["enc"], s["emb"], s["pos"], B.TRAINED, s["status"])
        B.merge_tokens_bwd(s["d_emb"], s["d_enc"], s["pos"], B.TRAINED, s["status"])
        return [s["emb"], s["d_enc"]]
    w = s["w"]
    plan = B.seg_plan(w.patch_counts, s["mode"]).to_device()
    B.encoder_fwd(s["x"], s["y"], s["layers"], s["heads"], s["ffn"], plan, w.softmax_scale, LN_EPS, s["ws"], s["lse"],
                  s["status"], rope=s["rope"])
    if s["mode"] == B.FROZEN:
        return [s["y"]]
    s["bucket"].zero_()
    B.encoder_bwd(s["dy"], s["x"], s["dx"], s["layers"], s["grads"], s["heads"], s["ffn"], plan, w.softmax_scale, LN_EPS,
                  s["lse"], s["ws"], s["ws_bwd"], s["status"], rope=s["rope"])
    return [s["y"], s["lse"], s["dx"], s["bucket"]]


def work(case):
    """Inputs read once, outputs written once; 2 FLOPs per multiply-add of the contractions, nothing recomputed."""
    w = _workload(case)
    T, trained = w.total_tokens, case["trained"]
    if case["kind"] == "seam":
        return {"bytes": 2 * (4 * T * w.merge_hidden + 4 * T), "flops": 0}
    heads, head_dim = case.get("heads", w.n_heads), case.get("head_dim", w.head_dim)
    act = 2 * T * heads * head_dim                           # bytes of one [T, hidden] bf16 tensor
    attn = (14 if trained else 4) * heads * head_dim * w.sum_n2
    if case["kind"] == "step":
        nbytes = (8 * act + 4 * heads * T) if trained else 4 * act         # q, k, v, dO in; O, dQ, dK, dV and LSE out
        if w.merge_hidden is not None:
            reads = 0 if w.merge_hidden == heads * head_dim else 2 * T * w.merge_hidden
            nbytes += reads + 2 * T * w.merge_hidden + 4 * T
        return {"bytes": nbytes, "flops": attn}
    hidden, n = heads * head_dim, case["layers"]
    weights = 12 * hidden * hidden                           # qkv 3, output 1, MLP 4 + 4 (ffn = 4 hidden)
    nbytes = n * 2 * weights + 2 * act + (4 * T * head_dim if case["rope"] else 0)
    flops = n * ((3 if trained else 1) * 2 * T * weights + attn)
    if trained:
        nbytes += n * 4 * weights + 2 * act + n * 4 * heads * T            # fp32 gradients, dy, dx, LSE
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the difference from the same path in 64 bits on the same bf16 inputs (rounding of the stored bf16
    intermediates and results).  Attention: relative 2.1e-3 to 2.5e-3 in every output, largest difference 3.1e-2 of the
    value.  Encoder: relative 3.1e-3 after one layer, 5.9e-3 after four and 9.2e-3 after 24, largest 2.7e-2 and 6.8e-2."""
    if case["kind"] == "seam":
        return "exact"
    if case["kind"] == "step":
        return {"rel": 1e-2, "max": 0.13}
    depth = math.sqrt(case["layers"])
    return {"rel": min(0.012 * depth, 0.03), "max": min(0.12 * depth, 0.4)}
