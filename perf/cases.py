"""Performance cases of the frame-quantized linear layer: what a program that serves or
quantizes a model with this library has it do, through the public entry points.

A case is a dict of plain values; its "kind" says which entry points it goes through:

    forward     fq_linear_forward: one layer, any batch size, with or without the de-noising gain
                and the rounding of the activations in the frame domain
    group       fq_linear_forward_group over independent layers with tiled frame operands
    structured  fq_linear_forward_implicit_group, the frames in structured form
    rebuild     fq_reconstruct_weight, then fq_dense_forward with the rebuilt weight
    rtn         fq_coefficients, fq_quantize_rtn and fq_pack: a layer quantized round-to-nearest
    gptq        fq_gptq_hessian, fq_quantize_gptq and fq_pack: a layer quantized with calibration

Shapes are those of `workloads` (a 256 x 256 layer, the ViT-B/16 MLP, Llama-2-7B and 70B linear
layers; rho = 16, k = ceil(r d / rho)).  Frames are real rotated (k, 16, d) tight fusion frames,
written out here with torch so that inputs and exact results need nothing from the library; the
codes of the forward cases are the round-to-nearest codes of Gaussian coefficients, which is
what the rotated frames make of trained weights.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_06082_gb300 as fq

RHO = 16


# ------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest layer, a few tokens: launch and dependency latency
        dict(name="layer256_m8", kind="forward", M=8, d_in=256, d_out=256, r_num=9, r_den=8,
             gamma=False, act_bits=0, outliers=False),
        # single-stream decode, one attention projection of a 7B model
        dict(name="7b_o_m1", kind="forward", M=1, d_in=4096, d_out=4096, r_num=11, r_den=10,
             gamma=False, act_bits=0, outliers=True),
        # batched decode: q|k|v of a 7B block in one launch
        dict(name="7b_qkv_group_m16", kind="group", layers=3, M=16, d_in=4096, d_out=4096,
             r_num=11, r_den=10, gamma=False, outliers=True),
        # continuous batching at a ragged batch size, the 7B down projection, filter on
        dict(name="7b_down_m40", kind="forward", M=40, d_in=11008, d_out=4096, r_num=11, r_den=10,
             gamma=True, act_bits=0, outliers=True),
        # the same block's gate|up with the frames in structured form
        dict(name="7b_gateup_structured_m16", kind="structured", layers=2, M=16, d_in=4096,
             d_out=11008, r_num=11, r_den=10, gamma=False, outliers=True),
        # a wide decode batch (or a short prompt) on a 70B projection
        dict(name="70b_q_m128", kind="forward", M=128, d_in=8192, d_out=8192, r_num=11, r_den=10,
             gamma=False, act_bits=0, outliers=True),
        # prefill of one 2048-token prompt, 7B gate, filter on
        dict(name="7b_gate_m2048", kind="forward", M=2048, d_in=4096, d_out=11008, r_num=11,
             r_den=10, gamma=True, act_bits=0, outliers=True),
        # ViT-B/16 MLP on 64 images of 197 tokens with 8-bit activations in the frame domain
        dict(name="vit_fc1_act8_m12608", kind="forward", M=12608, d_in=768, d_out=3072, r_num=11,
             r_den=10, gamma=False, act_bits=8, outliers=False),
        # the largest prefill: 4096 tokens through a 70B projection
        dict(name="70b_q_m4096", kind="forward", M=4096, d_in=8192, d_out=8192, r_num=11,
             r_den=10, gamma=False, act_bits=0, outliers=True),
        # the weight rebuilt for prefill-heavy serving, then a 2048-token batch through it
        dict(name="7b_q_rebuild_m2048", kind="rebuild", M=2048, d_in=4096, d_out=4096, r_num=11,
             r_den=10, gamma=True, outliers=True),
        # quantizing a 7B projection without calibration data
        dict(name="7b_q_rtn", kind="rtn", d_in=4096, d_out=4096, r_num=11, r_den=10),
        # quantizing ViT-B/16 fc1 with 1024 calibration tokens
        dict(name="vit_fc1_gptq", kind="gptq", d_in=768, d_out=3072, r_num=11, r_den=10,
             tokens=1024, clip=True),
    ]


_SHAPES = ((256, 256), (768, 3072), (3072, 768), (4096, 4096), (4096, 11008), (11008, 4096),
           (8192, 8192))
_REDUNDANCY = ((1, 1), (11, 10), (11, 10), (9, 8), (6, 5))


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _dim(rng, lo, hi):
    """A multiple of 16 with a reasonably square factor pair, over the logarithm of the range."""
    while True:
        d = 16 * _log_int(rng, lo // 16, hi // 16)
        a, b = _factor_pair(d)
        if b <= 16 * a:
            return d


def _shape(rng, lo, hi):
    if rng.random() < 0.5:
        fits = [s for s in _SHAPES if max(s) <= hi and min(s) >= lo]
        if fits:
            return rng.choice(fits)
    return _dim(rng, lo, hi), _dim(rng, lo, hi)


def draw(rng):
    cost = {c["kind"]: 0.0 for c in listed()}
    for c in listed():
        cost[c["kind"]] = max(cost[c["kind"]], work(c)["flops"])
    kind = rng.choices(("forward", "group", "structured", "rebuild", "rtn", "gptq"),
                       (50, 14, 12, 10, 7, 7))[0]
    while True:
        r_num, r_den = rng.choice(_REDUNDANCY)
        c = dict(kind=kind, r_num=r_num, r_den=r_den)
        if kind == "gptq":
            c["d_in"], c["d_out"] = _shape(rng, 256, 3072)
            c.update(tokens=_log_int(rng, 128, 1024), clip=rng.random() < 0.5)
            if c["d_in"] > 768:
                continue
        elif kind == "rtn":
            c["d_in"], c["d_out"] = _shape(rng, 256, 4096)
        else:
            c["d_in"], c["d_out"] = _shape(rng, 256, 11008)
            c.update(gamma=rng.random() < 0.5, outliers=rng.random() < 0.5)
            if kind in ("group", "structured"):
                c.update(layers=rng.randint(2, 3), M=_log_int(rng, 1, 64))
            elif kind == "rebuild":
                c.update(M=_log_int(rng, 64, 4096))
            else:
                c.update(M=_log_int(rng, 1, 12608),
                         act_bits=rng.choice((0, 0, 0, 0, 0, 8, 8, rng.randint(2, 7))))
        if work(c)["flops"] <= cost[kind]:
            return c


# -------------------------------------------------------------------------------- the frames
def _factor_pair(d):
    a = math.isqrt(d)
    while d % a:
        a -= 1
    return a, d // a


def _k(case, d):
    return -(-case["r_num"] * d // (case["r_den"] * RHO))


def _sizes(case):
    d_in, d_out = case["d_in"], case["d_out"]
    return d_in, _k(case, d_in) * RHO, _k(case, d_out) * RHO, d_out


def _rotation(d, seed):
    """The random draws of a rotation: (a, b, gauss_a, gauss_b, perm, signs), host arrays."""
    a, b = _factor_pair(d)
    g = np.random.Generator(np.random.PCG64(seed))
    return (a, b, g.standard_normal((a, a)), g.standard_normal((b, b)),
            g.permutation(d).astype(np.int64), g.choice((-1.0, 1.0), d))


def _haar(gauss):
    q, r = np.linalg.qr(gauss)
    return q * np.sign(np.diag(r))


def _frame(k, d, rot, dtype):
    """Analysis operator (k * 16, d) of the rotated (k, 16, d) tight fusion frame: 8 disjoint
    runs of d / 16 complex coordinates, each modulated by k roots of unity and realified, then
    T = T_u R^T with R = Pi (Q_a kron Q_b) D."""
    dev = "cuda"
    a, b, ga, gb, perm, signs = rot
    w = d // RHO
    ki = torch.arange(k, device=dev)[:, None]
    T = torch.zeros(RHO * k, d, dtype=dtype, device=dev)
    for j in range(RHO // 2):
        q = torch.arange(j * w, (j + 1) * w, device=dev)[None, :]
        ang = ((ki * q) % k).double() * (2.0 * math.pi / k)
        re, im = torch.cos(ang) / math.sqrt(k), torch.sin(ang) / math.sqrt(k)
        block = T[2 * j * k:2 * (j + 1) * k, 2 * j * w:2 * (j + 1) * w].view(k, 2, w, 2)
        block[:, 0, :, 0] = re
        block[:, 0, :, 1] = im
        block[:, 1, :, 0] = -im
        block[:, 1, :, 1] = re
    T *= torch.from_numpy(signs).to(dev, dtype)
    Qa = torch.from_numpy(_haar(ga)).to(dev, dtype)
    Qb = torch.from_numpy(_haar(gb)).to(dev, dtype)
    T = torch.matmul(Qa, torch.matmul(T.view(-1, a, b), Qb.t()))
    return T.reshape(RHO * k, d)[:, torch.from_numpy(perm).to(dev)].contiguous()


# --------------------------------------------------------------------------------- the inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _tokens(g, M, d, outliers):
    x = torch.randn(M, d, generator=g, device="cuda")
    if outliers:               # the same 1% of channels large for every token
        ch = torch.randperm(d, generator=g, device="cuda")[:max(1, d // 100)]
        x[:, ch] *= 30.0
    return x.bfloat16()


def _codes(g, n_out, n_in, std):
    """Round-to-nearest codes, fp16 scale and zero, and gain of Gaussian coefficients."""
    C = torch.randn(n_out, n_in, generator=g, device="cuda") * std
    mn, mx = C.amin(1), C.amax(1)
    zero, scale = mn.half(), ((mx - mn) / 3).half()
    s, z = scale.float()[:, None], zero.float()[:, None]
    codes = torch.clamp(torch.round((C - z) / s), 0, 3).to(torch.uint8)
    P = C.square().mean(1)
    return codes, scale, zero, P / (P + scale.float().square() / 12)


def _layer_inputs(case, seed, layer):
    """Codes with their scale, zero and gain, and the two rotations, of one layer."""
    _, n_in, n_out, _ = _sizes(case)
    s = 1000003 * (seed + 1) + 101 * layer
    codes, scale, zero, gain = _codes(_generator(s), n_out, n_in, 0.02)
    return dict(codes=codes, scale=scale, zero=zero, gamma=gain if case["gamma"] else None,
                rot_in=_rotation(case["d_in"], [s, 1]), rot_out=_rotation(case["d_out"], [s, 2]))


def _operators(case, L):
    """Dense bf16 T_in and T_out^T of a layer."""
    d_in, n_in, n_out, d_out = _sizes(case)
    return (_frame(n_in // RHO, d_in, L["rot_in"], torch.float32).bfloat16(),
            _frame(n_out // RHO, d_out, L["rot_out"], torch.float32).t().contiguous().bfloat16())


def _input(case, seed):
    return _tokens(_generator(7919 * (seed + 1)), case["M"], case["d_in"], case["outliers"])


def _quantizer_inputs(case, seed):
    """Weight and frame operators (fp32 of an fp64 construction), and for the calibrated
    quantizer the fp64 coefficients and the tokens' frame representation."""
    d_in, n_in, n_out, d_out = _sizes(case)
    g = _generator(104729 * (seed + 1))
    W = torch.randn(d_out, d_in, generator=g, device="cuda") / math.sqrt(d_in)
    T_in = _frame(n_in // RHO, d_in, _rotation(d_in, [seed, 3]), torch.float64)
    T_out = _frame(n_out // RHO, d_out, _rotation(d_out, [seed, 4]), torch.float64)
    if case["kind"] == "rtn":
        return W, T_in.float(), T_out.float()
    C = T_out @ (W.double() @ T_in.t())
    A = torch.randn(case["tokens"], d_in, generator=g, device="cuda", dtype=torch.float64)
    A = A @ (torch.randn(d_in, d_in, generator=g, device="cuda", dtype=torch.float64)
             / math.sqrt(d_in) + torch.eye(d_in, device="cuda", dtype=torch.float64))
    return C.contiguous(), (A @ T_in.t()).contiguous()


# ---------------------------------------------------------------------------- prepare and run
def _zeros(nbytes):
    return torch.zeros(max(nbytes, 256), dtype=torch.uint8, device="cuda")


def _i16(n):
    return torch.empty(n, dtype=torch.int16, device="cuda")


def _pack(L, n_out, n_in):
    words = torch.empty(fq.fq_packed_words(n_out, n_in), dtype=torch.int32, device="cuda")
    return fq.fq_pack(L["codes"], L["scale"].view(torch.int16), L["zero"].view(torch.int16),
                      n_out, n_in, words)


def _tiled(T):
    rows, cols = T.shape
    out = _zeros(fq.fq_frame_tiles_bytes(rows, cols))
    fq.fq_frame_tile(T, rows, cols, out, out.numel())
    return out


def prepare(case, seed):
    kind = case["kind"]
    d_in, n_in, n_out, d_out = _sizes(case)
    st = dict(case=case)
    if kind == "rtn":
        st["W"], st["T_in"], st["T_out"] = _quantizer_inputs(case, seed)
        st["C"] = torch.empty(n_out, n_in, device="cuda")
        st["ws"] = _zeros(fq.fq_coefficients_workspace_bytes(d_out, n_in))
    elif kind == "gptq":
        st["C"], st["Z"] = _quantizer_inputs(case, seed)
        st["H"] = torch.empty(n_in, n_in, dtype=torch.float64, device="cuda")
        st["ws"] = _zeros(fq.fq_gptq_workspace_bytes(n_out, n_in))
    if kind in ("rtn", "gptq"):
        st["codes"] = torch.empty(n_out, n_in, dtype=torch.uint8, device="cuda")
        st["scale"], st["zero"] = _i16(n_out), _i16(n_out)
        st["gamma"] = torch.empty(n_out, device="cuda")
        st["words"] = torch.empty(fq.fq_packed_words(n_out, n_in), dtype=torch.int32,
                                  device="cuda")
        return st

    M = case["M"]
    x = st["x"] = _input(case, seed)
    ys = st["ys"] = [torch.empty(M, d_out, dtype=torch.bfloat16, device="cuda")
                     for _ in range(case.get("layers", 1))]
    Ls = [_layer_inputs(case, seed, i) for i in range(len(ys))]
    packs = [_pack(L, n_out, n_in) for L in Ls]
    gammas = [L["gamma"] for L in Ls]
    if kind == "structured":
        F_in = fq.fq_frame_implicit(n_in // RHO, RHO, d_in, Ls[0]["rot_in"])   # one input frame
        st["layers"] = [fq.ImplicitLayer(x, F_in, C,
                                         fq.fq_frame_implicit(n_out // RHO, RHO, d_out,
                                                              L["rot_out"]), g, y)
                        for L, C, g, y in zip(Ls, packs, gammas, ys)]
        st["ws"] = _zeros(fq.fq_implicit_group_workspace_bytes(M, st["layers"]))
        return st
    ops = [_operators(case, L) for L in Ls]
    if kind == "group":
        st["layers"] = [fq.Layer(x, d_in, T_in, C, T_out_t, d_out, g, y, _tiled(T_in),
                                 _tiled(T_out_t))
                        for (T_in, T_out_t), C, g, y in zip(ops, packs, gammas, ys)]
        st["ws"] = _zeros(fq.fq_group_workspace_bytes(M, st["layers"]))
        return st
    (st["T_in"], st["T_out_t"]), st["C"], st["gamma"] = ops[0], packs[0], gammas[0]
    if kind == "rebuild":
        st["W_hat"] = torch.empty(d_out, d_in, dtype=torch.bfloat16, device="cuda")
        st["ws"] = _zeros(fq.fq_reconstruct_workspace_bytes(d_in, n_in, n_out, d_out))
        st["ws_dense"] = _zeros(fq.fq_dense_workspace_bytes(M, d_in, d_out))
    else:
        st["mode"] = fq.FQ_BF16 | (fq.FQ_ACT_BITS(case["act_bits"]) if case["act_bits"] else 0)
        st["ws"] = _zeros(fq.fq_workspace_bytes(M, d_in, n_in, n_out, d_out, st["mode"]))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    d_in, n_in, n_out, d_out = _sizes(case)
    ws, nb = st["ws"], st["ws"].numel()
    if kind in ("rtn", "gptq"):
        C, codes, scale, zero, gamma = st["C"], st["codes"], st["scale"], st["zero"], st["gamma"]
        if kind == "rtn":
            fq.fq_coefficients(st["W"], d_out, d_in, st["T_in"], n_in, st["T_out"], n_out, C, ws,
                               nb)
            fq.fq_quantize_rtn(C, n_out, n_in, codes, scale, zero, gamma)
            first = C
        else:
            fq.fq_gptq_hessian(st["Z"], case["tokens"], n_in, st["H"])
            fq.fq_quantize_gptq(C, n_out, n_in, st["H"], codes, scale, zero, gamma, ws, nb,
                                clip=case["clip"])
            first = st["H"]
        P = fq.fq_pack(codes, scale, zero, n_out, n_in, st["words"])
        return [first, codes, scale, zero, gamma, P.words]
    M, x, ys = case["M"], st["x"], st["ys"]
    if kind == "structured":
        fq.fq_linear_forward_implicit_group(M, st["layers"], ws, nb)
    elif kind == "group":
        fq.fq_linear_forward_group(M, st["layers"], ws, nb)
    elif kind == "rebuild":
        fq.fq_reconstruct_weight(st["T_in"], st["C"], st["T_out_t"], d_in, d_out, st["gamma"],
                                 st["W_hat"], ws, nb)
        fq.fq_dense_forward(x, M, d_in, st["W_hat"], d_out, ys[0], st["ws_dense"],
                            st["ws_dense"].numel())
        return [st["W_hat"], ys[0]]
    else:
        fq.fq_linear_forward(x, M, d_in, st["T_in"], st["C"], st["T_out_t"], d_out, st["gamma"],
                             ys[0], ws, nb, st["mode"])
    return ys


# ------------------------------------------------------------------------------ work and exact
def work(case):
    d_in, n_in, n_out, d_out = _sizes(case)
    codes = n_out * n_in // 4 + 4 * n_out
    kind = case["kind"]
    if kind == "rtn":
        return {"bytes": 4 * (d_in * d_out + n_in * d_in + n_out * d_out + n_out * n_in + n_out)
                + n_out * n_in + codes,
                "flops": 2.0 * n_in * d_out * (d_in + n_out)}
    if kind == "gptq":
        return {"bytes": 8 * (n_out * n_in + case["tokens"] * n_in + n_in * n_in) + 4 * n_out
                + n_out * n_in + codes,
                "flops": 1.0 * n_in * n_in * (case["tokens"] + 2 * n_in / 3 + n_out)}
    M, gain = case["M"], 4 * n_out if case["gamma"] else 0
    io = 2 * M * (d_in + d_out)
    product = 2.0 * n_in * n_out
    if kind == "rebuild":
        return {"bytes": 2 * (n_in * d_in + n_out * d_out + d_in * d_out) + codes + gain + io,
                "flops": d_in * (product + 2.0 * n_out * d_out) + 2.0 * M * d_in * d_out}
    if kind == "structured":
        def frame(d):          # rotation factors, permutation and signs
            a, b = _factor_pair(d)
            return 4 * (a * a + b * b) + 8 * d

        def apply(n, d):       # the rotation, and the block-diagonal operator
            return 2.0 * d * sum(_factor_pair(d)) + 2.0 * n * d / (RHO // 2)
        g = case["layers"]
        return {"bytes": frame(d_in) + g * (frame(d_out) + codes + gain + 2 * M * d_out)
                + 2 * M * d_in,
                "flops": M * (apply(n_in, d_in) + g * (product + apply(n_out, d_out)))}
    layer = 2 * (n_in * d_in + n_out * d_out) + codes + gain
    flops = M * (product + 2.0 * (n_in * d_in + n_out * d_out))
    if kind == "group":
        g = case["layers"]
        return {"bytes": g * (layer + 2 * M * d_out) + 2 * M * d_in, "flops": g * flops}
    return {"bytes": layer + io, "flops": flops}


def _exact_forward(case, L, x, T_in, T_out_t, act_bits=0):
    z = x.double() @ T_in.double().t()
    delta = 1.0
    if act_bits:
        lim = 2 ** (act_bits - 1) - 1
        delta = z.abs().max() / lim
        z = torch.clamp(torch.round(z / delta), -lim, lim)
    u = (z @ L["codes"].double().t()) * L["scale"].double() \
        + z.sum(1, keepdim=True) * L["zero"].double()
    u *= delta
    if L["gamma"] is not None:
        u *= L["gamma"].double()
    return u @ T_out_t.double().t()


def exact(case, seed):
    kind = case["kind"]
    d_in, n_in, n_out, d_out = _sizes(case)
    if kind in ("rtn", "gptq"):
        if kind == "rtn":
            W, T_in, T_out = (t.double() for t in _quantizer_inputs(case, seed))
            first = C = T_out @ (W @ T_in.t())
        else:
            C, Z = _quantizer_inputs(case, seed)
            first = Z.t() @ Z
            if case["clip"]:
                mu, sd = C.mean(), C.std(correction=0)
                C = torch.clamp(C, mu - 2 * sd, mu + 2 * sd)
        scale = ((C.amax(1) - C.amin(1)) / 3).half().double()
        P = C.square().mean(1)
        return [first, None, None, None, P / (P + scale.square() / 12), None]
    x = _input(case, seed)
    out = []
    for i in range(case.get("layers", 1)):
        L = _layer_inputs(case, seed, i)
        if kind == "structured":
            if i == 0:
                T_in = _frame(n_in // RHO, d_in, L["rot_in"], torch.float64)
            T_out_t = _frame(n_out // RHO, d_out, L["rot_out"], torch.float64).t()
        else:
            T_in, T_out_t = _operators(case, L)
        if kind == "rebuild":
            g = L["gamma"].double() if L["gamma"] is not None else 1.0
            C = L["codes"].double() * L["scale"].double()[:, None] + L["zero"].double()[:, None]
            W = (T_out_t.double() * g) @ (C @ T_in.double())
            return [W, x.double() @ W.t()]
        out.append(_exact_forward(case, L, x, T_in, T_out_t, case.get("act_bits", 0)))
    return out
