"""Workloads of the Sigma-Delta-quantized linear layer, as a program that uses this package runs them.

A case is a dict of plain values; `op` says which part of the package's work it is:

  forward  y = layer(x) for the linears of a decoder layer (or one linear), one plan each, through
           `Plan.forward`; with `deterministic` through `sdq_prep_activations` + `sdq_contract`, the
           bit-reproducible pair that a program takes that needs the same bits from run to run
  encode   W (fp32) -> codes and scales (`Plan.encode`), packed for the contraction (`Plan.pack`)
  gptq     the same with GPTQ block compensation (`Plan.encode_gptq`), as a checkpoint is quantized
  save     a live layer's tiled codes -> plain -> base-3 bytes (`sdq_unpack`, `sdq_pack_base3`); binary
           codes are stored in the plain layout itself
  load     the way back: base-3 bytes -> plain -> tiled (`sdq_unpack_base3`, `sdq_pack`)

`linears` lists the plans of a case as "rows x inputs @ OSR", for instance "12288x4096@2;4096x4096@2".
Layers whose linears read the same input at one OSR (q/k/v, gate/up) are one plan over their rows, as
`workloads.shared_input_groups` forms them.

Ranges: batches of 1 to 4096 rows, inputs 512 to 28672, rows 200 to 57344 (odd ones among them), blocks 64 to
512, OSR 3/2 to 3, ternary and binary codes, both scale modes of the encoder.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

import paper_2510_03275_gb300 as P

LLAMA7B = "12288x4096@2;4096x4096@2;22016x4096@2;4096x11008@2"           # q/k/v, o, gate/up, down
LLAMA70B = "10240x8192@2;8192x8192@2;57344x8192@2;8192x28672@2"
LLAMA13B_MULTIOSR = "15360x5120@3/2;5120x5120@2;13824x5120@3/2;13824x5120@2;5120x13824@3"
OPT125M = "2304x768@5/2;768x768@5/2;3072x768@5/2;768x3072@5/2"           # q/k/v, o, fc1, fc2


def _forward(name, linears, m, block=128, ternary=True, deterministic=False):
    c = {"op": "forward", "linears": linears, "m": m, "block": block, "ternary": ternary,
         "deterministic": deterministic}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one small linear, one token: nothing but latency
        _forward("single-256x512-m1", "256x512@2", 1, block=512),
        # a small model's layer, 16 sequences decoding, 1-bit codes at a fractional OSR
        _forward("opt125m-layer-m16", OPT125M, 16, ternary=False),
        # one sequence decoding: the layer's codes are read once per token
        _forward("llama7b-layer-m1", LLAMA7B, 1),
        _forward("llama70b-layer-m1", LLAMA70B, 1),
        # 8 sequences decoding on a layer whose linears have their own OSRs
        _forward("llama13b-multiosr-m8", LLAMA13B_MULTIOSR, 8),
        # a serving batch of 64 sequences
        _forward("llama7b-layer-m64", LLAMA7B, 64),
        # a short prompt of odd length
        _forward("llama7b-layer-m201", LLAMA7B, 201),
        # a long prompt (or many): the largest call
        _forward("llama70b-layer-m4096", LLAMA70B, 4096),
        # quantizing a model: one linear without, one with calibration
        {"name": "encode-llama7b-gate", "op": "encode", "linears": "11008x4096@2", "block": 128, "ternary": True,
         "mean": False},
        {"name": "gptq-llama7b-q", "op": "gptq", "linears": "4096x4096@2", "block": 128, "ternary": True,
         "mean": False},
        # writing a checkpoint, and reading one
        {"name": "save-llama70b-gate", "op": "save", "linears": "28672x8192@2", "block": 128, "ternary": True},
        {"name": "load-llama70b-gate", "op": "load", "linears": "28672x8192@2", "block": 128, "ternary": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward"] * 6 + ["encode", "encode", "gptq", "save", "load"])
    block = rng.choice([128, 128, 128, 128, 64, 256, 512])
    osr = rng.choice(["2", "2", "2", "3/2", "5/2", "3"])
    ternary = rng.random() < 0.75
    top_n, top_k = {"forward": (28672, 28672), "encode": (11008, 11008), "gptq": (4096, 4096),
                    "save": (28672, 8192), "load": (28672, 8192)}[op]
    n = _log_int(rng, 200, top_n)
    if rng.random() < 0.6:
        n = max(1, n // 128) * 128
    k = max(block, _log_int(rng, 512, top_k) // block * block)
    lin = f"{n}x{k}@{osr}"
    if op == "forward":
        # decode batches, prompts up to a few hundred tokens, long prompts
        lo, hi = rng.choice([(1, 4), (2, 64), (8, 64), (65, 767), (65, 767), (768, 4096)])
        return _forward(None, lin, _log_int(rng, lo, hi), block, ternary, rng.random() < 0.2)
    c = {"op": op, "linears": lin, "block": block, "ternary": ternary}
    if op in ("encode", "gptq"):
        c["mean"] = rng.random() < 0.2
    return c


# ----------------------------------------------------------------- inputs
def _linears(case):
    out = []
    for s in case["linears"].split(";"):
        shape, osr = s.split("@")
        n, k = shape.split("x")
        out.append((int(n), int(k), Fraction(osr)))
    return out


def _desc(case, n, k, osr):
    return P.LayerDesc(n, k, case["block"], osr, P.SDQ_TERNARY if case["ternary"] else P.SDQ_BINARY, 1,
                       P.SDQ_ALPHA_MEANABS if case.get("mean") else P.SDQ_ALPHA_MAXABS)


def _signs(seed, i, block):
    return np.where(np.random.default_rng([seed, i, 500]).integers(0, 2, size=block) == 1, 1, -1).astype(np.int8)


def _gen(seed, i):
    g = torch.Generator(device="cuda")
    g.manual_seed(1009 * seed + i)
    return g


def _plain_codes(g, n, k_eff, ternary):
    """Random codes in the plain layout (int32 words): ternary ones with half of them 0, or signs."""
    bits = 2 if ternary else 1
    wpr = 4 * -(-k_eff * bits // 128)
    w = torch.randint(-2 ** 31, 2 ** 31, (n, wpr), generator=g, device="cuda", dtype=torch.int32)
    if ternary:
        s = torch.randint(-2 ** 31, 2 ** 31, (n, wpr), generator=g, device="cuda", dtype=torch.int32)
        w &= 0x55555555
        s &= w
        w |= s << 1
    full, rest = divmod(k_eff * bits, 32)
    if rest:
        w[:, full] &= (1 << rest) - 1
        full += 1
    w[:, full:] = 0
    return w.reshape(-1)


def _weights(g, n, k):
    """Student-t(5) weights of standard deviation 0.02, every row with a scale of its own."""
    z = torch.randn((n, k), generator=g, device="cuda")
    chi = torch.zeros_like(z)
    for _ in range(5):
        chi.addcmul_(*[torch.randn((n, k), generator=g, device="cuda")] * 2)
    z.div_(chi.div_(5).sqrt_()).mul_(0.02 / math.sqrt(5 / 3))
    return z.mul_(torch.exp2(torch.rand((n, 1), generator=g, device="cuda") * 2 - 1))


def _factor(g, k):
    """An upper-triangular factor with a positive diagonal, as of an inverse Hessian."""
    u = torch.triu(torch.randn((k, k), generator=g, device="cuda"), diagonal=1) * (0.1 / k ** 0.5)
    u.diagonal().copy_(torch.rand((k,), generator=g, device="cuda") + 0.5)
    return u


def prepare(case, seed):
    state = {"op": case["op"], "m": case.get("m"), "deterministic": case.get("deterministic"),
             "ternary": case["ternary"], "parts": []}
    for i, (n, k, osr) in enumerate(_linears(case)):
        g = _gen(seed, i)
        desc = _desc(case, n, k, osr)
        plan = P.Plan(desc, _signs(seed, i, case["block"]))
        part = {"plan": plan}
        if case["op"] == "forward":
            part["tiled"] = plan.pack(_plain_codes(g, n, plan.k_eff, case["ternary"]))
            part["alpha"] = 0.05 + 0.1 * torch.rand(n, generator=g, device="cuda")
            part["x"] = torch.randn((case["m"], k), generator=g, device="cuda").to(torch.bfloat16)
            part["ws"] = plan.alloc_workspace(case["m"])
        elif case["op"] in ("encode", "gptq"):
            part["w"] = _weights(g, n, k)
            if case["op"] == "gptq":
                part["u"] = _factor(g, k)
        else:
            plain = _plain_codes(g, n, plan.k_eff, case["ternary"])
            part["bad"] = torch.zeros(1, dtype=torch.int32, device="cuda")
            part["plain"] = torch.empty_like(plain)
            if case["ternary"]:
                part["base3"] = torch.empty(P.sdq_base3_bytes(desc), dtype=torch.uint8, device="cuda")
            if case["op"] == "save":
                part["tiled"] = plan.pack(plain)
            else:
                part["tiled"] = plan.alloc_tiled()
                if case["ternary"]:
                    P.sdq_pack_base3(plan.handle, plain, part["base3"])
                else:
                    part["plain"] = plain
        state["parts"].append(part)
    return state


# -------------------------------------------------------------- one pass
def run(state):
    out = []
    for p in state["parts"]:
        plan = p["plan"]
        if state["op"] == "forward":
            if state["deterministic"]:
                m = state["m"]
                y = torch.empty((m, plan.desc.n_out), dtype=torch.float32, device="cuda")
                P.sdq_prep_activations(plan.handle, p["x"], m, p["ws"])
                P.sdq_contract(plan.handle, p["tiled"], p["alpha"], m, y, p["ws"])
            else:
                y = plan.forward(p["tiled"], p["alpha"], p["x"], p["ws"])
            out.append(y)
        elif state["op"] in ("encode", "gptq"):
            codes, alpha = plan.encode(p["w"]) if state["op"] == "encode" else plan.encode_gptq(p["w"], p["u"])
            out += [codes, plan.pack(codes), alpha]
        elif state["op"] == "save":
            P.sdq_unpack(plan.handle, p["tiled"], p["plain"], p["bad"])
            if state["ternary"]:
                P.sdq_pack_base3(plan.handle, p["plain"], p["base3"])
            out += [p["plain"], p["base3"], p["bad"]] if state["ternary"] else [p["plain"], p["bad"]]
        else:
            if state["ternary"]:
                P.sdq_unpack_base3(plan.handle, p["base3"], p["plain"], p["bad"])
            P.sdq_pack(plan.handle, p["plain"], p["tiled"])
            out += [p["plain"], p["tiled"], p["bad"]]
    return out


# ------------------------------------------------- what a pass cannot do without
def work(case):
    by = fl = 0
    for n, k, osr in _linears(case):
        k_eff = int(k * osr)
        plain = n * (4 * (-(-k_eff * (2 if case["ternary"] else 1) // 128))) * 4
        if case["op"] == "forward":
            m = case["m"]
            by += plain + 4 * n + 2 * m * k + 4 * m * n
            # the shorter of the two orders: codes times upsampled x, or rebuilt weights times x
            fl += min(2 * m * n * k_eff + 2 * m * k_eff * case["block"],
                      2 * m * n * k + 2 * n * k_eff * case["block"])
        elif case["op"] in ("encode", "gptq"):
            by += 4 * n * k + 2 * plain + 4 * n
            fl += 2 * n * k_eff * case["block"]
            if case["op"] == "gptq":
                by += 2 * k * k
                fl += n * k * k + 2 * n * k_eff * case["block"]
        else:
            base3 = n * 16 * -(-(-(-k_eff // 5)) // 16) if case["ternary"] else 0
            by += 2 * plain + base3
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Codes, scales and stored bytes are exact. Outputs: up to 4 batch rows the activations enter with 18 bits
    below their group's largest, up to 16 with 12, above with 9 (the rounding of bf16): measured against `exact`
    over these ranges 4.7e-6, 2.5e-4 and 2.0e-3, stated at about four times that."""
    if case["op"] != "forward":
        return "exact"
    return {"rel": 2e-5 if case["m"] <= 4 else 1e-3 if case["m"] <= 16 else 8e-3}


# ------------------------------------------------------------ in 64 bits
def _resample_matrix(n_in, n_to):
    """The band-limited resampler n_in -> n_to (n_to x n_in), from the transforms of the unit vectors."""
    if n_in == n_to:
        return torch.eye(n_in, dtype=torch.float64, device="cuda")
    spec = torch.fft.fft(torch.eye(n_in, dtype=torch.float64, device="cuda"), dim=0)
    b = min(n_in, n_to)
    out = torch.zeros((n_to, n_in), dtype=torch.complex128, device="cuda")
    out[:b // 2] = spec[:b // 2]
    out[n_to - b // 2 + 1:] = spec[n_in - b // 2 + 1:]
    if n_to > n_in:      # the highest frequency is shared by its two places
        out[b // 2] += spec[b // 2] / 2
        out[n_to - b // 2] += spec[b // 2] / 2
    else:                # ... or folded from them
        out[b // 2] += spec[b // 2] + spec[n_in - b // 2]
    return torch.fft.ifft(out, dim=0).real * (n_to / n_in)


def _hadamard(block, signs):
    h = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    while h.shape[0] < block:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return torch.as_tensor(signs.astype(np.float64), device="cuda")[:, None] * h / math.sqrt(block)


def _codes64(plain, n, k_eff, ternary):
    bits = 2 if ternary else 1
    w = plain.reshape(n, -1)
    sh = torch.arange(0, 32, bits, device="cuda", dtype=torch.int32)
    f = (w[:, :, None] >> sh) & (2 ** bits - 1)
    v = torch.where(f == 3, -1.0, f.double()) if ternary else 2.0 * f.double() - 1.0
    return v.reshape(n, -1)[:, :k_eff].double()


def exact(case, seed):
    if case["op"] in ("save", "load"):
        return None
    out, block = [], case["block"]
    for i, (n, k, osr) in enumerate(_linears(case)):
        g, n_b, nblk = _gen(seed, i), int(block * osr), k // block
        had = _hadamard(block, _signs(seed, i, block))
        if case["op"] == "forward":
            plain = _plain_codes(g, n, nblk * n_b, case["ternary"]).reshape(n, -1)
            alpha = (0.05 + 0.1 * torch.rand(n, generator=g, device="cuda")).double()
            x = torch.randn((case["m"], k), generator=g, device="cuda").to(torch.bfloat16).double()
            back = _resample_matrix(n_b, block).T @ had.T          # n_b x block: codes of a block -> its weights
            y = torch.empty((case["m"], n), dtype=torch.float64, device="cuda")
            for r in range(0, n, 2048):
                c = _codes64(plain[r:r + 2048], min(2048, n - r), nblk * n_b, case["ternary"])
                w = (c.reshape(-1, n_b) @ back).reshape(-1, k)
                y[:, r:r + 2048] = (x @ w.T) * alpha[r:r + 2048]
            out.append(y)
            continue
        w = _weights(g, n, k)
        up = _resample_matrix(block, n_b) @ had.T                  # n_b x block
        alpha = torch.empty(n, dtype=torch.float64, device="cuda")
        for r in range(0, n, 1024):
            v = (w[r:r + 1024].double().reshape(-1, nblk, block) @ up.T).abs()
            alpha[r:r + 1024] = v.mean(dim=(1, 2)) if case["mean"] else v.amax(dim=(1, 2))
        out += [None, None, alpha]
    return out
