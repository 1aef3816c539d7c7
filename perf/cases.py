"""Performance cases of the quantised linear layer: the calls a training or serving program makes, and their sizes.

A case is one pass over one or several linear layers ("linears": "COUNTxOUTxIN,...") of one of five kinds:

  block_ap   forward and backward with the fake-quantised latent weight (W, s and z are trained)
  e2e_qp     forward, input gradient and step-size gradient on packed codes (s, or s and z, are trained)
  forward    packed-weight forward alone: decoding one or a few sequences, batched decoding, prompts
  export     round-to-nearest quantisation of a weight: s and z from each group's range, codes packed, and unpacked again
  weight     fake quantiser and its straight-through backward on their own, for a program with contractions of its own

"group" 0 stands for one group per row (channel-wise quantisation).  Weights are Student-t (heavy tails), one input
channel in a hundred ten times larger; activations N(0, 1); gradients N(0, 0.01^2); step sizes of the trained kinds lie a
few per cent off the min/max grid they started from.
"""
from __future__ import annotations

import torch

import paper_2407_11062_b200.binding as eqat

BLOCK_7B = "4x4096x4096,2x11008x4096,1x4096x11008"
BLOCK_13B = "4x5120x5120,2x13824x5120,1x5120x13824"
BLOCK_70B = "2x8192x8192,2x1024x8192,2x28672x8192,1x8192x28672"

MAX_FLOPS = 2.0e13            # most arithmetic of a drawn case: that of the largest listed one


def _case(name, kind, linears, bits, group, tokens=0, zero_points="u8"):
    return {"name": name, "kind": kind, "linears": linears, "bits": bits, "group": group, "tokens": tokens,
            "zero_points": zero_points}


def listed():
    return [
        # training one block's linears with fake-quantised weights
        _case("train_512_w2g64", "block_ap", "1x512x512", 2, 64, 256),                      # smallest: unit tests, toy models
        _case("train_7b_block_w4g128", "block_ap", BLOCK_7B, 4, 128, 4096),                 # batch 2 x context 2048
        _case("train_4096_w4_channel", "block_ap", "1x4096x4096", 4, 0, 1777),              # channel-wise, ragged batch
        # end-to-end training of the step sizes on frozen codes
        _case("tune_7b_block_w2g64", "e2e_qp", BLOCK_7B, 2, 64, 16384),                     # batch 4 x context 4096; the largest
        _case("tune_13b_up_w3g128", "e2e_qp", "1x13824x5120", 3, 128, 8192),                # 3-bit stream, batch 4 x 2048
        _case("tune_7b_down_w4g64_fp16z", "e2e_qp", "1x4096x11008", 4, 64, 1531, "fp16"),   # s and z trained, short ragged batch
        # inference on packed codes
        _case("decode_1_7b_block_w2g64", "forward", BLOCK_7B, 2, 64, 1),                    # one sequence
        _case("decode_8_70b_block_w4g128", "forward", BLOCK_70B, 4, 128, 8),                # eight sequences, large model
        _case("decode_40_13b_block_w3g128", "forward", BLOCK_13B, 3, 128, 40),              # batched serving
        _case("prompt_333_7b_block_w2g64", "forward", BLOCK_7B, 2, 64, 333),                # a prompt of ordinary length
        # weight passes
        _case("export_7b_block_w2g64", "export", BLOCK_7B, 2, 64),                          # hand-off of a block
        _case("weight_70b_up_w2g64", "weight", "1x28672x8192", 2, 64),
    ]


def _log_uniform(rng, low, high):
    return low * (high / low) ** rng.random()


def draw(rng):
    kind = rng.choice(["block_ap", "e2e_qp", "forward", "forward", "forward", "export", "weight"])
    out = 64 * int(round(_log_uniform(rng, 8, 448)))
    inp = 128 * int(round(_log_uniform(rng, 4, 224)))
    bits = rng.choice([2, 2, 3, 4])
    groups = [64, 64, 128, 128, 32, 0] + ([256] if inp % 256 == 0 else [])
    case = {"kind": kind, "linears": "%dx%dx%d" % (rng.choice([1, 1, 2, 3]), out, inp), "bits": bits,
            "group": rng.choice(groups), "tokens": 0, "zero_points": "u8"}
    if kind in ("block_ap", "e2e_qp"):
        case["tokens"] = int(round(_log_uniform(rng, 100, 16384)))
    elif kind == "forward":
        case["tokens"] = int(round(_log_uniform(rng, 1, 4096)))
    if kind in ("e2e_qp", "forward") and rng.random() < 0.25:
        case["zero_points"] = "fp16"
    while work(case)["flops"] > MAX_FLOPS:
        case["tokens"] = case["tokens"] * 2 // 3
    return case


def _shapes(case):
    shapes = []
    for part in case["linears"].split(","):
        count, out, inp = (int(v) for v in part.split("x"))
        shapes += [(out, inp)] * count
    return shapes


def _group(case, inp):
    return case["group"] or inp


# ------------------------------------------------------------------ what a program holds before the call
def _normal(gen, shape, std):
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).bfloat16()


def _weight(gen, out, inp):
    n = torch.randn((out, inp), generator=gen, device="cuda", dtype=torch.float32)
    u = torch.rand((2, out, inp), generator=gen, device="cuda", dtype=torch.float32).clamp_(min=1e-6)
    n.div_(torch.sqrt_(torch.log_(u[0].mul_(u[1])).mul_(-0.5)))             # chi-square(4) / 4 = -ln(u v) / 2
    gain = torch.ones(inp, device="cuda")
    gain[torch.randperm(inp, generator=gen, device="cuda")[: (inp + 99) // 100]] = 10.0
    return n.mul_(0.02).mul_(gain).bfloat16()


def _empty(shape, dtype):
    return torch.empty(shape, device="cuda", dtype=dtype)


def _linear(case, gen, out, inp):
    kind, bits, tokens = case["kind"], case["bits"], case["tokens"]
    group = _group(case, inp)
    zp = eqat.EQAT_ZP_FP16 if case["zero_points"] == "fp16" else eqat.EQAT_ZP_U8
    plain = eqat.make_desc(bits, group, out, inp, tokens)
    groups = (out, inp // group)
    W = _weight(gen, out, inp)
    s, z = _empty(groups, torch.float32), _empty(groups, torch.float32)
    L = {"desc": eqat.make_desc(bits, group, out, inp, tokens, zero_point_format=zp)}
    packed = {"Wq_packed": _empty((out, inp * bits // 8), torch.uint8), "z8": _empty(groups, torch.uint8),
              "s16": _empty(groups, torch.float16)}
    if kind == "export":
        return dict(L, W=W, s=s, z=z, codes=_empty((out, inp), torch.uint8), **packed)
    eqat.eqat_minmax_init(plain, W, s, z)
    s.mul_(1.0 + 0.03 * torch.randn(groups, generator=gen, device="cuda"))
    if kind == "weight":
        return dict(L, W=W, s=s, z=z, dW_hat=_normal(gen, (out, inp), 1e-2), W_hat=_empty((out, inp), torch.bfloat16),
                    dW=_empty((out, inp), torch.bfloat16), ds=_empty(groups, torch.float32), dz=_empty(groups, torch.float32))
    L["X"], L["Y"] = _normal(gen, (tokens, inp), 1.0), _empty((tokens, out), torch.bfloat16)
    if kind != "forward":
        L["dY"], L["dX"] = _normal(gen, (tokens, out), 1e-2), _empty((tokens, inp), torch.bfloat16)
        L["ds"] = _empty(groups, torch.float32)
        L["dz"] = _empty(groups, torch.float32) if kind == "block_ap" or zp == eqat.EQAT_ZP_FP16 else None
        op = eqat.EQAT_OP_FAKEQUANT_BWD if kind == "block_ap" else eqat.EQAT_OP_PACKED_BWD_DS
        scratch = eqat.workspace_bytes(L["desc"], op)
        L["workspace"] = _empty((scratch,), torch.uint8) if scratch else None
    if kind == "block_ap":
        return dict(L, W=W, s=s, z=z, W_hat=_empty((out, inp), torch.bfloat16), dW=_empty((out, inp), torch.bfloat16))
    eqat.eqat_quantize_pack(plain, W, s, z, packed["Wq_packed"], packed["z8"], packed["s16"])
    L["Wq_packed"], L["s16"] = packed["Wq_packed"], packed["s16"]
    L["z"] = packed["z8"]
    if zp == eqat.EQAT_ZP_FP16:
        L["z"] = (L["z"].float() + 0.1 * torch.randn(groups, generator=gen, device="cuda")).half()
    return L


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"kind": case["kind"], "linears": [_linear(case, gen, out, inp) for out, inp in _shapes(case)]}


# ------------------------------------------------------------------ one pass
_RESULTS = {"block_ap": ("Y", "W_hat", "dX", "dW", "ds", "dz"), "e2e_qp": ("Y", "dX", "ds", "dz"), "forward": ("Y",),
            "export": ("s", "z", "Wq_packed", "z8", "s16", "codes"), "weight": ("W_hat", "dW", "ds", "dz")}


def run(state):
    kind, linears = state["kind"], state["linears"]
    if kind == "block_ap" and len(linears) > 1:
        eqat.eqat_block_ap_step(linears)
    elif kind == "e2e_qp" and len(linears) > 1:
        eqat.eqat_e2e_qp_step(linears)
    else:
        for L in linears:
            if kind == "block_ap":
                eqat.qlinear_fakequant_fwd(L["desc"], L["X"], L["W"], L["s"], L["z"], L["Y"], L["W_hat"])
                eqat.qlinear_fakequant_bwd(L["desc"], L["X"], L["dY"], L["W"], L["s"], L["z"], L["W_hat"], L["dX"], L["dW"],
                                           L["ds"], L["dz"], L["workspace"])
            elif kind == "e2e_qp":
                eqat.qlinear_packed_fwd(L["desc"], L["X"], L["Wq_packed"], L["s16"], L["z"], L["Y"])
                eqat.qlinear_packed_bwd_dx(L["desc"], L["dY"], L["Wq_packed"], L["s16"], L["z"], L["dX"])
                eqat.qlinear_packed_bwd_ds(L["desc"], L["X"], L["dY"], L["Wq_packed"], L["z"], L["s16"], L["ds"], L["dz"],
                                           L["workspace"])
            elif kind == "forward":
                eqat.qlinear_packed_fwd(L["desc"], L["X"], L["Wq_packed"], L["s16"], L["z"], L["Y"])
            elif kind == "export":
                eqat.eqat_minmax_init(L["desc"], L["W"], L["s"], L["z"])
                eqat.eqat_quantize_pack(L["desc"], L["W"], L["s"], L["z"], L["Wq_packed"], L["z8"], L["s16"])
                eqat.eqat_unpack(L["desc"], L["Wq_packed"], L["codes"])
            else:
                eqat.eqat_fakequant_weight(L["desc"], L["W"], L["s"], L["z"], L["W_hat"])
                eqat.eqat_ste_bwd(L["desc"], L["dW_hat"], L["W"], L["s"], L["z"], L["dW"], L["ds"], L["dz"])
    return [L[name] for L in linears for name in _RESULTS[kind] if L[name] is not None]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind, bits, T = case["kind"], case["bits"], case["tokens"]
    zbytes = 2 if case["zero_points"] == "fp16" else 1
    nbytes = flops = 0
    for out, inp in _shapes(case):
        n, groups = out * inp, out * (inp // _group(case, inp))
        codes = n * bits // 8 + groups * (2 + zbytes)
        if kind == "block_ap":                       # W, s, z, X, dY in; Y, W_hat, dX, dW, ds, dz out
            nbytes += 6 * n + 16 * groups + 4 * T * (out + inp)
            flops += 6 * T * n
        elif kind == "e2e_qp":                       # codes, s, z, X, dY in; Y, dX, ds (dz) out
            nbytes += codes + 4 * groups * zbytes + 4 * T * (out + inp)
            flops += 6 * T * n
        elif kind == "forward":
            nbytes += codes + 2 * T * (out + inp)
            flops += 2 * T * n
        elif kind == "export":                       # W in; s, z, packed codes, z8, s16, unpacked codes out
            nbytes += 2 * n + 11 * groups + n * bits // 8 + n
        else:                                        # W, s, z, dW_hat in; W_hat, dW, ds, dz out
            nbytes += 8 * n + 16 * groups
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "export":
        return "exact"                               # codes, packed bytes, and s and z of one group each
    if case["kind"] == "weight":
        return {"rel": 1e-6, "max": 5e-6}            # fp32 group sums in another order (seen against fp64: 1.3e-7, 1.3e-6)
    # bf16 results, W_hat rounded to bf16 or not (seen against fp64: 2.4e-3; largest 1.5e-2 in Y, 5.7e-2 in the dX of
    # outlier channels' neighbours)
    return {"rel": 1e-2, "max": 6e-2 if case["kind"] == "forward" else 0.2}


# ------------------------------------------------------------------ the same results in 64 bits
def _unpacked(packed, bits):
    runs = packed.view(packed.shape[0], -1, bits).to(torch.int64)                      # eight codes in `bits` bytes
    value = sum(runs[..., i] << (8 * i) for i in range(bits))
    shifts = torch.arange(0, 8 * bits, bits, device=packed.device)
    return ((value[..., None] >> shifts) & ((1 << bits) - 1)).reshape(packed.shape[0], -1)


def _exact_linear(kind, L):
    d = L["desc"]
    out, inp, group = d.out_features, d.in_features, d.group

    def groups(v):
        return v.view(out, inp // group, group)

    if kind in ("block_ap", "weight"):
        s, zr, Q = L["s"][..., None], torch.round(L["z"])[..., None], float((1 << d.bits) - 1)
        r = torch.round(groups(L["W"].float()) / s)                                    # the code is decided in 32 bits
        p = r + zr
        inside, c = (p >= 0) & (p <= Q), p.clamp(0, Q) - zr
        W_hat = (c.double() * s.double()).view(out, inp)
        partial = torch.where(inside, r.double() - groups(L["W"].double()) / s.double(), c.double())
        G = L["dW_hat"].double() if kind == "weight" else L["dY"].double().t() @ L["X"].double()
        results = {"W_hat": W_hat, "dW": (groups(G) * inside).view(out, inp), "ds": (groups(G) * partial).sum(-1),
                   "dz": (groups(G) * torch.where(inside, 0.0, -s.double())).sum(-1)}
    else:
        codes = _unpacked(L["Wq_packed"], d.bits)
        step, centred = L["s16"].double()[..., None], groups(codes.double()) - L["z"].double()[..., None]
        W_hat, results = (centred * step).view(out, inp), {}
        if kind == "e2e_qp":
            G = groups(L["dY"].double().t() @ L["X"].double())
            results = {"ds": (G * centred).sum(-1), "dz": -step[..., 0] * G.sum(-1)}
    if kind != "weight":
        results["Y"] = L["X"].double() @ W_hat.t()
    if kind in ("block_ap", "e2e_qp"):
        results["dX"] = L["dY"].double() @ W_hat
    return [results[name] for name in _RESULTS[kind] if L[name] is not None]


def exact(case, seed):
    if case["kind"] == "export":
        return None                                  # compared bit for bit
    state = prepare(case, seed)
    return [v for L in state["linears"] for v in _exact_linear(state["kind"], L)]
