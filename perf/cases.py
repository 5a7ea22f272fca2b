"""The workloads whose speed counts: what a program built on this package has it do, through the public entry points.

Twelve listed cases and a generator of further ones over the same ranges.  Sizes are those of `workloads.CONFIGS`
(16 heads, d' = 16, d_v 64 for the 360M layer, 112 / 128 for the 1.3B layer), of the benchmark and of the tests.
Inputs are seeded normals with the scales of `workloads.CONFIGS`, made on the device.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what the caller has before the call
    run(state)          one pass
    work(case)          bytes and operations that a pass cannot do without
    tolerance(case)     how far another correct implementation may be off
"""
import math

import torch

import paper_2402_18668_b200 as based
from paper_2402_18668_b200.autograd import linear_attention
from paper_2402_18668_b200.generation import DecodeGraph

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # interactive generation of one stream: one token through one layer's recurrent mixer, latency is all
        dict(name="decode_one_stream", kind="decode", B=1, H=16, d_v=128, dtype="bf16"),
        # a small serving batch, both mixers of a token as one replayed graph on the compact (153-row) state
        dict(name="generation_graph", kind="graph", B=16, H=16, d_v=128, window=64, sym=True, dtype="bf16"),
        # a full serving batch with sequences of unequal lengths, eager calls: the recurrent, the window and the
        # convolution mixer's step of one token (the generation configuration's batch)
        dict(name="serving_token", kind="serve", B=128, H=16, d_v=128, window=64, C=8192, width=3, dtype="bf16"),
        # a few ragged prompt pieces appended to sequences in flight (1.3B model's true head width, compact state)
        dict(name="prompt_piece", kind="prefill", B=3, H=16, L=777, d_feat=16, d_v=112, dtype="bf16", state="continue_sym", scale=1.0),
        # prompts of the 360M model's layer, outputs only (scoring)
        dict(name="prefill_360m", kind="prefill", B=4, H=16, L=2048, d_feat=16, d_v=64, dtype="bf16", state="none", scale=0.25),
        # prompts of the 1.3B model's layer before generation: outputs and state
        dict(name="prefill_1p3b", kind="prefill", B=8, H=16, L=4096, d_feat=16, d_v=128, dtype="bf16", state="new", scale=0.25),
        # long context: both attention mixers over 32k tokens
        dict(name="mixer_pair_32k", kind="pair", B=2, H=16, L=32768, d_v=64, window=64, dtype="bf16"),
        # one training step's share of the 360M layer: forward and backward under autograd
        dict(name="train_360m", kind="train", B=4, H=16, L=2048, d_v=64, dtype="bf16"),
        # a small fp32 check run: the prompt of a tiny model with its state
        dict(name="prefill_tiny_f32", kind="prefill", B=1, H=2, L=256, d_feat=16, d_v=64, dtype="f32", state="new", scale=1.0),
        # training in fp32 (no mixed precision): forward and backward under autograd
        dict(name="train_f32", kind="train", B=2, H=16, L=1024, d_v=64, dtype="f32"),
        # the feature-dimension ablation (d' other than 16), outputs and state
        dict(name="prefill_dfeat24", kind="prefill", B=4, H=16, L=2048, d_feat=24, d_v=64, dtype="bf16", state="new", scale=0.25),
        # the gated convolution over a whole batch of sequences
        dict(name="baseconv_layer", kind="conv", B=8, N=4096, C=8192, width=3, dtype="bf16"),
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, even over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "graph", "serve", "piece", "prefill", "prefill", "pair", "train", "prefill_f32", "train_f32",
                       "dfeat", "conv"])
    H = rng.choice([2, 8, 12, 16, 16, 25, 32])
    d_v = rng.choice([64, 112, 128])
    window = rng.choice([16, 48, 64, 64, 100, 128])
    if kind == "decode":
        return dict(kind="decode", B=_log(rng, 1, 32), H=H, d_v=d_v, dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "graph":
        return dict(kind="graph", B=_log(rng, 1, 64), H=H, d_v=d_v, window=window, sym=rng.random() < 0.7, dtype="bf16")
    if kind == "serve":
        return dict(kind="serve", B=_log(rng, 8, 128), H=rng.choice([8, 12, 16]), d_v=d_v, window=window,
                    C=8 * _log(rng, 64, 1024), width=rng.choice([2, 3, 4]), dtype="bf16")
    if kind == "piece":
        return dict(kind="prefill", B=_log(rng, 1, 16), H=H, L=_log(rng, 16, 2048), d_feat=16, d_v=d_v, dtype="bf16",
                    state=rng.choice(["continue", "continue_sym"]), scale=1.0)
    if kind == "prefill":
        B = _log(rng, 1, 8)
        return dict(kind="prefill", B=B, H=H, L=_log(rng, 64, max(1024, min(32768, 524288 // (B * H)))), d_feat=16, d_v=d_v,
                    dtype="bf16", state=rng.choice(["none", "new"]), scale=0.25)
    if kind == "pair":
        return dict(kind="pair", B=_log(rng, 1, 2), H=rng.choice([8, 12, 16]), L=_log(rng, 4096, 32768), d_v=64, window=window,
                    dtype="bf16")
    if kind == "train":
        return dict(kind="train", B=_log(rng, 1, 8), H=rng.choice([8, 12, 16]), L=_log(rng, 256, 4096), d_v=d_v, dtype="bf16")
    if kind == "prefill_f32":
        return dict(kind="prefill", B=_log(rng, 1, 4), H=rng.choice([2, 8, 16]), L=_log(rng, 32, 1024), d_feat=16, d_v=d_v,
                    dtype="f32", state=rng.choice(["none", "new", "continue"]), scale=1.0)
    if kind == "train_f32":
        return dict(kind="train", B=_log(rng, 1, 2), H=rng.choice([2, 8, 16]), L=_log(rng, 64, 1024), d_v=64, dtype="f32")
    if kind == "dfeat":
        return dict(kind="prefill", B=_log(rng, 1, 4), H=rng.choice([8, 12, 16]), L=_log(rng, 128, 2048),
                    d_feat=rng.choice([8, 24, 32]), d_v=d_v, dtype="bf16", state=rng.choice(["none", "new"]), scale=0.25)
    return dict(kind="conv", B=_log(rng, 1, 8), N=_log(rng, 64, 4096), C=8 * _log(rng, 64, 1024), width=rng.choice([2, 3, 4]),
                dtype=rng.choice(["bf16", "bf16", "f32"])) if rng.random() < 0.7 else \
        dict(kind="conv", B=8, N=_log(rng, 64, 2048), C=4096, width=3, dtype="f32")


# ---------------------------------------------------------------------------------------------- inputs
def _phi(x, d):
    """The feature map: 1, x / d^(1/4), x (x) x / (sqrt 2 sqrt d)."""
    x = x.float()
    o = torch.einsum("...m,...n->...mn", x, x).flatten(-2) / (math.sqrt(2.0) * math.sqrt(d))
    return torch.cat([torch.ones_like(x[..., :1]), x * d ** -0.25, o], dim=-1)


def _sequence_state(rnd, B, H, d, d_v, sym, tokens=128):
    """The state that a prompt of random keys and values leaves: what a sequence in flight carries."""
    f = _phi(rnd(B * H, tokens, d), d)
    kv = torch.bmm(f.transpose(1, 2), rnd(B * H, tokens, d_v)).view(B, H, -1, d_v)
    z = f.sum(1).view(B, H, -1)
    if sym:                                  # one row per unordered pair: sqrt 2 off the diagonal
        m, n = torch.triu_indices(d, d, device=DEV)
        w = torch.where(m == n, 1.0, math.sqrt(2.0)).to(DEV)
        kv = torch.cat([kv[:, :, :1 + d], kv[:, :, 1 + d + m * d + n] * w[:, None]], dim=2)
        z = torch.cat([z[:, :, :1 + d], z[:, :, 1 + d + m * d + n] * w], dim=2)
    return kv.contiguous(), z.contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    dt = DTYPES[case["dtype"]]

    def rnd(*shape, scale=1.0, dtype=torch.float32):
        t = torch.randn(*shape, generator=g, device=DEV)
        return (t * scale).to(dtype) if scale != 1.0 else t.to(dtype)

    s = dict(case=case, kind=case["kind"])
    kind, B = case["kind"], case["B"]
    if kind in ("decode", "serve", "graph"):
        H, d_v = case["H"], case["d_v"]
        s["kv"], s["z"] = _sequence_state(rnd, B, H, 16, d_v, case.get("sym", False))
        s["q"], s["k"], s["v"] = rnd(B, H, 16, dtype=dt), rnd(B, H, 16, dtype=dt), rnd(B, H, d_v, dtype=dt)
        if kind != "decode":
            w = case["window"]
            s["qw"], s["kw"], s["vw"] = (rnd(B, H, 64, dtype=dt) for _ in range(3))
            s["kc"], s["vc"] = rnd(B, H, w, 64, dtype=dt), rnd(B, H, w, 64, dtype=dt)
        if kind == "serve":
            C, width = case["C"], case["width"]
            s["pos"] = torch.randint(0, 2048, (B,), generator=g, device=DEV, dtype=torch.int32)
            s["a"], s["g"] = rnd(B, C, dtype=dt), rnd(B, C, dtype=dt)
            s["h"], s["b2"] = rnd(width, C, scale=0.5), rnd(C, scale=0.1)
            s["conv_state"] = rnd(B, width - 1, C, dtype=dt)
        if kind == "graph":
            s["graph"] = DecodeGraph(s["kv"], s["z"], s["kc"], s["vc"], pos=1000 + seed % 100, dtype=dt, sym=case["sym"])
    elif kind in ("prefill", "pair", "train"):
        H, L, d, d_v, scale = case["H"], case["L"], case.get("d_feat", 16), case["d_v"], case.get("scale", 1.0)
        if kind == "train":
            scale = 0.25
        s["q"], s["k"] = rnd(B, H, L, d, scale=scale, dtype=dt), rnd(B, H, L, d, scale=scale, dtype=dt)
        s["v"] = rnd(B, H, L, d_v, dtype=dt)
        if kind == "pair":
            s["qw"], s["kw"] = rnd(B, H, L, 64, dtype=dt), rnd(B, H, L, 64, dtype=dt)
        if kind == "train":
            s["dout"] = rnd(B, L, H * d_v, dtype=dt)
            for n in "qkv":
                s[n].requires_grad_(True)
        state = case.get("state", "none")
        if state == "new":
            s["kv"], s["z"] = based.new_state(B, H, d_v, DEV, d_feat=d)
        elif state != "none":
            s["kv"], s["z"] = _sequence_state(rnd, B, H, d, d_v, state == "continue_sym")
        s["flags"] = {"continue": based.BASED_STATE_CONTINUE,
                      "continue_sym": based.BASED_STATE_CONTINUE | based.BASED_STATE_SYM}.get(state, based.BASED_STATE_ZERO_INIT)
    elif kind == "conv":
        N, C, width = case["N"], case["C"], case["width"]
        s["a"], s["g"] = rnd(B, N, C, dtype=dt), rnd(B, N, C, dtype=dt)
        s["h"], s["b2"] = rnd(width, C, scale=0.5), rnd(C, scale=0.1)
    return s


# ---------------------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "decode":
        return based.based_decode_step(s["q"], s["k"], s["v"], s["kv"], s["z"]), s["kv"], s["z"]
    if kind == "graph":
        out, out_w = s["graph"].step(s["q"], s["k"], s["v"], s["qw"], s["kw"], s["vw"])
        return out, out_w, s["kv"], s["z"], s["kc"], s["vc"]
    if kind == "serve":
        out = based.based_decode_step(s["q"], s["k"], s["v"], s["kv"], s["z"])
        out_w = based.swa_decode_step_ragged(s["qw"], s["kw"], s["vw"], s["kc"], s["vc"], s["pos"])
        out_c = based.baseconv_gate_step(s["a"], s["g"], s["h"], s["b2"], s["conv_state"])
        return out, out_w, out_c, s["kv"], s["z"], s["kc"], s["vc"], s["conv_state"]
    if kind == "prefill":
        if "kv" not in s:
            return based.based_prefill(s["q"], s["k"], s["v"])
        return based.based_prefill(s["q"], s["k"], s["v"], kv_state=s["kv"], z_state=s["z"], flags=s["flags"]), s["kv"], s["z"]
    if kind == "pair":
        return (based.based_prefill(s["q"], s["k"], s["v"]),
                based.swa_forward(s["qw"], s["kw"], s["v"], window=s["case"]["window"]))
    if kind == "train":
        # the heads side by side, as the layer's output projection takes them and its gradient comes back
        out = linear_attention(s["q"], s["k"], s["v"]).transpose(1, 2).reshape(s["dout"].shape)
        return (out.detach(),) + torch.autograd.grad(out, (s["q"], s["k"], s["v"]), s["dout"])
    return based.baseconv_gate_forward(s["a"], s["g"], s["h"], s["b2"])


# ---------------------------------------------------------------------------------------------- accounting
def work(case):
    kind, B, e = case["kind"], case["B"], 2 if case["dtype"] == "bf16" else 4
    if kind == "conv":
        n = B * case["N"] * case["C"]
        return {"bytes": 3 * n * e + (case["width"] + 1) * case["C"] * 4, "flops": n * (2 * case["width"] + 6)}
    BH, d_v, d = B * case["H"], case["d_v"], case.get("d_feat", 16)
    pairs = 1 + d + d * (d + 1) // 2         # distinct features: one per unordered pair
    if kind in ("decode", "serve", "graph"):
        rows = pairs if case.get("sym") else 1 + d + d * d
        w = {"bytes": BH * (2 * rows * (d_v + 1) * 4 + (2 * d + 2 * d_v) * e), "flops": BH * 4 * rows * (d_v + 1)}
        if kind != "decode":                 # cache read, new slot, q, k, v, out
            w["bytes"] += BH * 64 * e * (2 * case["window"] + 6)
            w["flops"] += BH * 4 * 64 * case["window"]
        if kind == "serve":                  # a, g, out, the state read and written
            w["bytes"] += B * case["C"] * e * (3 + 2 * (case["width"] - 1))
            w["flops"] += B * case["C"] * (2 * case["width"] + 6)
        return w
    L = case["L"]
    T = BH * L
    rows = pairs if case.get("state") == "continue_sym" else 1 + d + d * d
    states = {"none": 0, "new": 1}.get(case.get("state", "none"), 2)
    n_bytes = T * (2 * d + 2 * d_v) * e + states * BH * rows * (d_v + 1) * 4
    # the cheaper of the quadratic and the chunked recurrent form (64-token chunks)
    flops = min(T * (L + 1) * (d + d_v), T * (4 * pairs * d_v + 128 * (d + d_v)))
    if states and flops < T * 2 * pairs * d_v:
        flops += T * 2 * pairs * d_v
    if kind == "pair":
        n_bytes += T * 3 * 64 * e
        flops += T * 4 * 64 * min(case["window"], L)
    if kind == "train":                      # forward as above; backward: q, k, v, out, dout in, three gradients out
        n_bytes += T * (4 * d + 4 * d_v) * e
        flops += min(T * (L + 1) * (5 * d + 3 * d_v), T * (10 * pairs * d_v + 128 * (5 * d + 3 * d_v)))
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    """Rounding only: about four times the distance to the same path in 64-bit arithmetic.  Measured on these cases and
    on drawn ones: bf16 results of the whole-sequence paths 2.3e-3 to 2.5e-3 (operands and results rounded to bf16), of
    the one-token steps and the convolution 1.6e-3 to 2.0e-3 (results rounded once); fp32 1e-7 to 8e-7 (sums of up to a
    few thousand terms)."""
    if case["dtype"] == "f32":
        return {"rel": 4e-6}
    return {"rel": 1e-2 if case["kind"] in ("train", "prefill", "pair") else 8e-3}
