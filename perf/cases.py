"""The work this library is used for, as cases that can be timed: the routed sparse attention of one transformer layer.

A case is one layer's pass on one GPU, through the binding's public entry points:

  train   gate projection (if the case has one), router + selection, forward, backward, gate backward
  infer   gate projection (if the case has one), router + selection, forward

Sizes are the repository's configurations and benchmark rows (latent grids of 480p and 720p video, 61 and 121 frames,
the 2048-token clip, the smallest grid of the tests), with the head counts of a whole model or of one GPU's share of one.
Inputs have the structure of `paper_2609_32882_b200.inputs` ("locality": smooth noise on the grid plus white noise), drawn
on the GPU.
"""
import math

import numpy as np
import torch

from paper_2609_32882_b200 import binding as vb

SEQ, ROW, BUDGET = vb.PER_SEQUENCE, vb.PER_QUERY, vb.PER_QUERY_BUDGET
BUDGET_LO, BUDGET_HI = 16, 256


def _case(name, kind, grid, heads_q, heads_kv, topk, *, mode=SEQ, batch=1, dim=128, wide=False, text=0, hidden=0,
          shared=False, f32=False):
    """One layer's pass.  grid: latent frames, rows, columns; topk: KV cubes kept per query cube (budget cases: unused);
    wide: cubes of 4x4x8 instead of 4x4x4 tokens; text: text tokens behind the video; hidden: width of the gate
    projection's input, 0 = the gate is handed in; shared: one block map per KV group; f32: outputs in fp32."""
    t, h, w = grid
    return {"name": name, "kind": kind, "t": t, "h": h, "w": w, "heads_q": heads_q, "heads_kv": heads_kv, "topk": topk,
            "mode": mode, "batch": batch, "dim": dim, "wide": wide, "text": text, "hidden": hidden, "shared": shared,
            "f32": f32}


def listed():
    return [
        # the smallest call: a toy grid as unit tests and bring-up of a training loop use it; launches and host time
        _case("tiny_train_d64", "train", (4, 8, 8), 2, 2, 2, mode=ROW, dim=64),
        # a 2048-token clip (low-resolution pre-training, distillation previews), per-query TopK, with its gate projection
        _case("clip_train", "train", (8, 16, 16), 12, 12, 8, mode=ROW, hidden=1536),
        # the same kind of clip served in a batch of two, ragged in every dimension
        _case("clip_infer_ragged", "infer", (9, 30, 45), 12, 12, 16, batch=2, hidden=1536),
        # 480p training with grouped query heads, 1/8 of the KV cubes per query
        _case("480p_train_gqa", "train", (21, 30, 52), 12, 3, 78, mode=ROW),
        # 480p serving with one block map per KV group
        _case("480p_infer_shared_map", "infer", (21, 30, 52), 12, 3, 78, mode=ROW, shared=True),
        # an odd grid with 64-channel heads and fp32 gradients (gradient checks, small models)
        _case("odd_train_d64_f32", "train", (13, 27, 47), 16, 16, 24, dim=64, f32=True),
        # 720p training of a whole 40-head layer: the repository's benchmark step
        _case("720p_train", "train", (21, 45, 80), 40, 40, 64),
        # 720p serving at top-128 with heads sharded over four GPUs, the gate projected from the full hidden state
        _case("720p_infer_top128", "infer", (21, 45, 80), 10, 10, 128, hidden=5120),
        # 720p with joint text tokens, heads sharded over eight GPUs, training with the gate projection
        _case("720p_train_text", "train", (21, 45, 80), 5, 5, 64, text=512, hidden=5120),
        # 720p training with a budget of 16..256 cubes per query cube, grouped heads
        _case("720p_train_budget", "train", (21, 45, 80), 8, 2, 0, mode=BUDGET),
        # 61 latent frames of 720p with cubes of 128 tokens: long-video training, heads sharded over two GPUs
        _case("220k_train_wide", "train", (61, 45, 80), 10, 10, 64, wide=True),
        # 121 latent frames of 720p with cubes of 128 tokens: long-video serving
        _case("436k_infer_wide", "infer", (121, 45, 80), 10, 10, 64, wide=True, hidden=2560),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: clips to long videos, training and serving, every option of the listed ones."""
    cap = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(["train", "infer"])
        wide = rng.random() < 0.3
        t, h, w = _log_int(rng, 4, 121), _log_int(rng, 8, 45), _log_int(rng, 8, 80)
        dim = 64 if rng.random() < 0.25 else 128
        heads_kv = _log_int(rng, 1, 40)
        rep = rng.choice([1, 1, 1, 2, 4])
        mode = rng.choice([SEQ, SEQ, ROW, BUDGET])
        n = _cubes(t, h, w, wide)
        topk = 0 if mode == BUDGET else _log_int(rng, min(8, n), max(min(8, n), min(128, n)))
        text = rng.choice([0, 0, 0, rng.randint(17, 600)])
        shared = rep > 1 and mode != BUDGET and rng.random() < 0.5
        c = _case("", kind, (t, h, w), heads_kv * rep, heads_kv, topk, mode=mode, batch=rng.choice([1, 1, 2]), dim=dim,
                  wide=wide, text=text, hidden=rng.choice([0, 8 * rng.randint(32, 640)]), shared=shared,
                  f32=rng.random() < 0.2)
        del c["name"]
        if c["heads_q"] > 40 or c["batch"] * c["heads_q"] * dim * t * h * w > 40 * 128 * 75600:
            continue
        if work(c)["flops"] <= cap:
            return c


def _cubes(t, h, w, wide):
    return -(-t // 4) * -(-h // 4) * -(-w // (8 if wide else 4))


def _smoothing(n, device):
    """Gaussian filter of sigma 2, truncated at 8, reflecting at both ends, as an n x n matrix."""
    taps = np.exp(-0.5 * (np.arange(-8, 9) / 2.0) ** 2)
    taps /= taps.sum()
    m = np.zeros((n, n), dtype=np.float32)
    for i in range(n):
        for k, c in zip(range(i - 8, i + 9), taps):
            k %= 2 * n
            m[i, k if k < n else 2 * n - 1 - k] += c
    return torch.from_numpy(m).to(device)


def _video(gen, batch, heads, t, h, w, dim, text, smooth):
    """[batch, heads, t*h*w + text, dim] bf16: unit-variance smooth noise + 0.3 white noise; text rows white."""
    out = torch.empty(batch, heads, t * h * w + text, dim, dtype=torch.bfloat16, device="cuda")
    for b in range(batch):
        for i in range(heads):
            x = torch.randn(t, h * w * dim, generator=gen, device="cuda")
            x = (smooth[0] @ x).view(t, h, w * dim)
            x = torch.matmul(smooth[1], x).view(t * h, w, dim)
            x = torch.matmul(smooth[2], x).view(t * h * w, dim)
            x = x / x.std() + 0.3 * torch.randn(t * h * w, dim, generator=gen, device="cuda")
            out[b, i, :t * h * w] = x
            if text:
                out[b, i, t * h * w:] = torch.randn(text, dim, generator=gen, device="cuda")
    return out


def prepare(case, seed):
    """Inputs of one pass on the GPU and the handle (maps, saved state, workspaces) a layer keeps."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    b, hq, hk, dim, text = case["batch"], case["heads_q"], case["heads_kv"], case["dim"], case["text"]
    grid = (case["t"], case["h"], case["w"])
    n_tok = grid[0] * grid[1] * grid[2]
    smooth = [_smoothing(n, "cuda") for n in grid]
    s = {"kind": case["kind"], "hidden": case["hidden"], "budgets": None}
    s["q"] = _video(gen, b, hq, *grid, dim, text, smooth)
    s["k"] = _video(gen, b, hk, *grid, dim, text, smooth)
    s["v"] = _video(gen, b, hk, *grid, dim, text, smooth)
    nnz_cap = 0
    if case["mode"] == BUDGET:
        n = _cubes(*grid, case["wide"])
        s["budgets"] = torch.randint(BUDGET_LO, BUDGET_HI + 1, (b, hq, n), generator=gen, device="cuda", dtype=torch.int32)
        nnz_cap = int(s["budgets"].clamp(max=n).sum(dim=-1).max())
    params = vb.make_params(b, hq, hk, dim, grid, cube=(4, 4, 8) if case["wide"] else (4, 4, 4), select_mode=case["mode"],
                            topk=case["topk"], out_dtype=vb.F32 if case["f32"] else vb.BF16, nnz_cap=nnz_cap,
                            text_len=text, flags=vb.FLAG_GROUP_ROUTING if case["shared"] else 0)
    s["attn"] = vb.Vsa2Attention(params)
    if case["hidden"]:
        s["x"] = torch.randn(b, n_tok, case["hidden"], generator=gen, device="cuda", dtype=torch.bfloat16)
        s["w_g"] = (torch.randn(case["hidden"], hq, generator=gen, device="cuda") * 0.5 / math.sqrt(case["hidden"])).bfloat16()
    else:
        s["gate"] = torch.tanh(0.5 * torch.randn(b, hq, n_tok, generator=gen, device="cuda"))
    if case["kind"] == "train":
        s["d_o"] = torch.randn(s["q"].shape, generator=gen, device="cuda", dtype=torch.bfloat16)
        if case["hidden"]:
            s["ws_gate"] = torch.empty(vb.vsa2_gate_bwd_workspace_bytes(params, case["hidden"]), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    attn, q, k, v, hidden = state["attn"], state["q"], state["k"], state["v"], state["hidden"]
    gate = state.get("gate")
    if hidden:
        x, w_g = state["x"], state["w_g"]
        gate = torch.empty(x.shape[0], w_g.shape[1], x.shape[1], dtype=torch.float32, device=x.device)
        vb.vsa2_gate_fwd(attn.p, hidden, x, w_g, gate)
    attn.route(q, k, state["budgets"])
    o, lse = attn.forward(q, k, v, gate)
    out = {"o": o, "lse": lse}
    if hidden:
        out["gate"] = gate
    if state["kind"] == "train":
        out["dq"], out["dk"], out["dv"], out["dgate"] = attn.backward(q, k, v, gate, o, lse, state["d_o"])
        if hidden:
            out["d_w_g"] = torch.empty(w_g.shape, dtype=torch.float32, device=x.device)
            out["dx"] = torch.empty(x.shape, dtype=attn.out_torch_dtype, device=x.device)
            vb.vsa2_gate_bwd(attn.p, hidden, x, w_g, gate, out["dgate"], out["d_w_g"], out["dx"], state["ws_gate"])
    return out


def work(case):
    """Bytes: every input once, every output once.  Operations: router scores (sub-cubes of 8 tokens), coarse attention,
    attention over the kept tokens and the text, gate projection; a backward pass has 2.5 times its forward's products."""
    b, hq, hk, dim, text = case["batch"], case["heads_q"], case["heads_kv"], case["dim"], case["text"]
    train, hidden = case["kind"] == "train", case["hidden"]
    n_tok = case["t"] * case["h"] * case["w"]
    n = _cubes(case["t"], case["h"], case["w"], case["wide"])
    rows = n_tok + text
    keep = sum(min(k, n) for k in range(BUDGET_LO, BUDGET_HI + 1)) / (BUDGET_HI - BUDGET_LO + 1) if case["mode"] == BUDGET else min(case["topk"], n)
    pairs = keep / n * n_tok * n_tok + text * (2 * n_tok + text)
    out = 4 if case["f32"] else 2
    q_bytes, kv_bytes, gate_bytes = b * hq * rows * dim, 2 * b * hk * rows * dim, 4 * b * hq * n_tok
    x_elems, w_elems = b * n_tok * hidden, hidden * hq
    nbytes = 2 * (q_bytes + kv_bytes) + out * q_bytes + 4 * b * hq * rows + gate_bytes + 2 * (x_elems + w_elems)
    flops = 4 * b * hq * dim * pairs * (3.5 if train else 1)
    flops += 4 * b * hq * dim * n * n * (3.5 if train else 1)
    flops += 2 * b * hq * dim * (n_tok / 8) ** 2
    flops += 2 * x_elems * hq * (3 if train else 1)
    if train:
        nbytes += 2 * q_bytes + out * (q_bytes + kv_bytes) + gate_bytes + out * x_elems + 4 * w_elems
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Largest relative error of an output between correct implementations with 16-bit operands.  Measured between the
    library's own forms (P and dS rounded once to bf16, to fp16, or carried as bf16 pairs; coarse branch in TF32 or bf16; the
    grid mirrored, which reverses the order of every sum): at most 2.6e-3 for o, dq, dk, dv and dgate, 3.7e-3 for dx and
    d_w_g; single elements up to 0.27 of the larger of their own value and the tensor's root mean square (dk of cubes that
    many queries keep)."""
    return {"rel": 1e-2, "max": 0.5}
