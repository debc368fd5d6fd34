"""Timed workloads of the BiGLA library: what a program around a ViG token mixer has it do.

A case names what is done ("do"), the sizes B (images), H (heads), L (tokens, or the patch grid Hh x Ww), dk and dv (head
sizes), the element type and the mean of the gate logits (0: fast decay, 2: slow decay, long memory).  Four things are done:

  infer   the mixer from its gate logits, vig_bigla_fwd_gates_bf16: the forward pass of a deployed model
  layer   the 2-D gating locality injection around it: vig_dwconv3x3, then vig_bigla_fwd_blend_bf16
  train   one training step of the mixer: gate preparation, forward, gradient, gradient through the gate preparation
  host    the mixer on pinned host buffers, vig_bigla_fwd_host

Values are those of the library's synthetic configurations: q, k, v, d_out ~ N(0, 1) with q scaled by dk^-0.5, gate logits
~ N(gate_mean, 1).
"""
import math

import torch

import paper_2405_18425_b200 as vig

TAU = 16.0
DK, DV = (16, 24, 32), (32, 48, 64)
HEADS = (2, 3, 4, 6, 12, 24)


def _case(name, do, B, H, L, dk, dv, dtype="bf16", gate_mean=0.0, Hh=0, Ww=0):
    return {"name": name, "do": do, "B": B, "H": H, "L": L, "dk": dk, "dv": dv, "dtype": dtype, "gate_mean": gate_mean, "Hh": Hh, "Ww": Ww}


def listed():
    return [
        # one photo through a ViG-T block: the latency of a single small call
        _case("infer_t224_one_image", "infer", 1, 4, 196, 24, 48),
        # the ordinary evaluation batches at 224 x 224
        _case("infer_t224", "infer", 128, 4, 196, 24, 48),
        _case("infer_b224", "infer", 64, 12, 196, 32, 64, gate_mean=2.0),
        # images that are not square: 240 x 320 pixels, 15 x 20 patches, ragged against every tile
        _case("infer_240x320", "infer", 24, 6, 300, 32, 64),
        # high resolution: 1024 x 1024 and 2048 x 2048
        _case("infer_t1024", "infer", 8, 4, 4096, 24, 48),
        _case("infer_t2048", "infer", 2, 4, 16384, 24, 48),
        # a block with the locality injection, as a deployed ViG-B runs it
        _case("layer_b224", "layer", 64, 12, 196, 32, 64, gate_mean=2.0, Hh=14, Ww=14),
        # training: the last stage of the hierarchical model (7 x 7 patches), ViG-B at 224, ViG-T at 1024
        _case("train_h_stage4", "train", 16, 24, 49, 16, 32),
        _case("train_b224", "train", 64, 12, 196, 32, 64, gate_mean=2.0),
        _case("train_t1024", "train", 8, 4, 4096, 24, 48),
        # full-precision training of a small batch (validating a run, debugging a loss)
        _case("train_s224_f32", "train", 8, 6, 196, 32, 64, dtype="f32"),
        # a caller whose activations live in host memory
        _case("host_b224", "host", 64, 12, 196, 32, 64, gate_mean=2.0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any of the things done, token counts from a single small image up to the listed batches."""
    do = rng.choice(("infer", "infer", "layer", "train", "train", "train_f32", "host"))
    H, dk, dv = rng.choice(HEADS), rng.choice(DK), rng.choice(DV)
    f32 = do == "train_f32"
    Hh = Ww = 0
    if do == "layer":
        Hh, Ww = rng.randint(5, 40), rng.randint(5, 40)
        L = Hh * Ww
    else:
        L = _log_uniform(rng, 25, 784 if f32 else 16384)
    # token-heads of the pass: the listed full batches have about 131 K to 151 K
    rows = _log_uniform(rng, 784, 9408 if f32 else 131072)
    B = max(1, min(256, rows // (H * L)))
    while H > 2 and B * H * L > (9408 if f32 else 131072):
        H //= 2
    case = _case("", "train" if f32 else do, B, H, L, dk, dv, dtype="f32" if f32 else "bf16", gate_mean=rng.choice((0.0, 2.0)), Hh=Hh, Ww=Ww)
    del case["name"]
    return case


def prepare(case, seed):
    do, B, H, L, dk, dv = (case[k] for k in ("do", "B", "H", "L", "dk", "dv"))
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    rng = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape, scale=1.0, mean=0.0):
        return (torch.randn(*shape, generator=rng, device="cuda") * scale + mean).to(dtype)

    s = {
        "do": do,
        "dtype": dtype,
        "q": normal(B, H, L, dk, scale=dk ** -0.5),
        "k": normal(B, H, L, dk),
        "v": normal(B, H, L, dv),
        "g_f": normal(B, H, L, dk, mean=case["gate_mean"]),
        "g_b": normal(B, H, L, dk, mean=case["gate_mean"]),
    }
    s["out"] = torch.empty_like(s["v"])
    if do == "host":
        for name in ("q", "k", "v", "g_f", "g_b", "out"):
            on_host = torch.empty(s[name].shape, dtype=dtype, pin_memory=True)
            s[name] = on_host.copy_(s[name])
    if do == "layer":
        C = H * dv
        s["x"] = normal(B, case["Hh"], case["Ww"], C)
        s["w"], s["bias"] = normal(C, 3, 3, scale=0.3), normal(C, scale=0.3)
        s["conv"] = torch.empty_like(s["x"])
        # the convolution's output laid out per head and its projection: products of the model's own dense layers
        s["o_local"], s["z"] = normal(B, H, L, dv), normal(B, H, L, dv)
    if do == "train":
        s["d_out"] = normal(B, H, L, dv)
        for name, like in (("la_f", "q"), ("la_b", "q"), ("dq", "q"), ("dk", "q"), ("dv", "v"), ("dg_f", "q"), ("dg_b", "q")):
            s[name] = torch.empty_like(s[like])
    return s


def run(s):
    do = s["do"]
    if do == "infer":
        return vig.vig_bigla_fwd_gates_bf16(s["q"], s["k"], s["v"], s["g_f"], s["g_b"], s["out"], TAU)
    if do == "host":
        return vig.vig_bigla_fwd_host(s["q"], s["k"], s["v"], s["g_f"], s["g_b"], s["out"], TAU)
    if do == "layer":
        vig.vig_dwconv3x3(s["x"], s["w"], s["bias"], s["conv"])
        vig.vig_bigla_fwd_blend_bf16(s["q"], s["k"], s["v"], s["g_f"], s["g_b"], s["o_local"], s["z"], s["out"], TAU)
        return s["conv"], s["out"]
    if s["dtype"] == torch.float32:
        vig.vig_gate_prep_f32(s["g_f"], s["g_b"], s["la_f"], s["la_b"], TAU)
        vig.vig_bigla_fwd_f32(s["q"], s["k"], s["v"], s["la_f"], s["la_b"], s["out"])
    else:
        vig.vig_gate_prep_bf16(s["g_f"], s["g_b"], s["la_f"], s["la_b"], TAU)
        vig.vig_bigla_fwd_bf16(s["q"], s["k"], s["v"], s["la_f"], s["la_b"], s["out"])
    # the gradients of the log gates turn into those of the gate logits in place
    vig.vig_bigla_bwd(s["q"], s["k"], s["v"], s["la_f"], s["la_b"], s["d_out"], s["dq"], s["dk"], s["dv"], s["dg_f"], s["dg_b"])
    vig.vig_gate_prep_bwd(s["g_f"], s["g_b"], s["dg_f"], s["dg_b"], s["dg_f"], s["dg_b"], TAU)
    return s["out"], s["dq"], s["dk"], s["dv"], s["dg_f"], s["dg_b"]


def work(case):
    do, dk, dv = case["do"], case["dk"], case["dv"]
    n = case["B"] * case["H"] * case["L"]
    elem = 4 if case["dtype"] == "f32" else 2
    # forward: q, k, both gates and v in, out; per direction a rank-one update of the dk x dv state and a product with it
    width, flops = 4 * dk + 2 * dv, 8 * dk * dv
    if do == "layer":
        # the two blend operands; the convolution's image in and out, nine multiply-adds an element
        width, flops = width + 4 * dv, flops + 18 * dv
    if do == "train":
        # d_out in, five gradients out; two walks of ten multiply-adds an element of the state
        width, flops = width + 4 * dk + 2 * dv, flops + 20 * dk * dv
    return {"bytes": width * elem * n, "flops": flops * n}


def tolerance(case):
    # fp32: sums of a few thousand fp32 products.  bf16: operands and results of 8 significant bits; single elements that
    # cancel are off by a few rounding steps of the largest terms.
    return {"rel": 1e-5, "max": 2e-4} if case["dtype"] == "f32" else {"rel": 1e-2, "max": 0.15}
