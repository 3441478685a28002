"""The calls that users of the library make, as measurable cases.

A case is a dict of plain values; its "kind" names the pattern of calls:

  forward   one quantised linear layer on device buffers (the operator itself)
  host      the same with activations in pinned host memory (the end-to-end entry)
  block     the seven projections of one decoder block, one call each, in the order a model runs them
  finetune  one layer's step of multiplicative fine-tuning: y, dx, dB and dA with the codes fixed
  qat       one layer's step of quantisation-aware training: codes of the current weight, their
            transpose, y, dx and the straight-through gradients dW, dB, dA
  quantize  the code-assignment step of the offline refinement (one layer's weight)

m = out-features, n = in-features, r = rank, M = tokens, bits = code width.  Inputs follow the recipe of
the package's `inputs` module (uniform codes, positive factors, normal activations, 1 % outlier columns
from 256 tokens on), drawn on the GPU.
"""
import math

import torch

from paper_2601_22716_b200 import binding as lords
from paper_2601_22716_b200 import inputs

GROUP = {2: 4, 3: 32, 4: 2}          # n is a multiple of the pack group
_ready = []
_books = {}


def listed():
    return [
        # the smallest call (the tiny configuration): what one call costs however little it computes
        dict(name="tiny_m4", kind="forward", m=256, n=256, r=4, M=4, bits=4),
        # the headline configuration: one token through a 4096 x 4096 projection
        dict(name="decode_q_m1", kind="forward", m=4096, n=4096, r=32, M=1, bits=4),
        # the same for a program whose activations live in host memory
        dict(name="decode_q_host_m1", kind="host", m=4096, n=4096, r=32, M=1, bits=4),
        # one token of text generation through a decoder block, 4-bit attention and 3-bit MLP (mixed widths)
        dict(name="block_m1_mixed", kind="block", h=4096, kv=1024, ffn=14336, M=1, bits=4, mlp_bits=3, r=32, r_kv=16, r_mlp=48),
        # a batch of eight sequences decoding together, all layers 4-bit
        dict(name="block_m8_nf4", kind="block", h=4096, kv=1024, ffn=14336, M=8, bits=4, mlp_bits=4, r=32, r_kv=16, r_mlp=32),
        # a prompt of 512 tokens through a block
        dict(name="block_m512_nf4", kind="block", h=4096, kv=1024, ffn=14336, M=512, bits=4, mlp_bits=4, r=32, r_kv=16, r_mlp=32),
        # a long prompt through the widest reduction, activation outliers included (compute-bound prefill)
        dict(name="prefill_down_m2048", kind="forward", m=4096, n=14336, r=32, M=2048, bits=4),
        # nothing a multiple of a tile: a short prompt, an odd hidden width, a rank from the small-rank table
        dict(name="ragged_m37", kind="forward", m=1000, n=2730, r=10, M=37, bits=4),
        # the finest scales the interface offers (parameter parity with blocks of 16), a batch of 16
        dict(name="rank128_m16", kind="forward", m=4096, n=4096, r=128, M=16, bits=4),
        # fine-tuning B and A of one projection on 512 tokens
        dict(name="finetune_q_m512", kind="finetune", m=4096, n=4096, r=32, M=512, bits=4),
        # quantisation-aware training of one projection on 1024 tokens
        dict(name="qat_q_m1024", kind="qat", m=4096, n=4096, r=32, M=1024, bits=4),
        # code assignment of the widest layer, 3 bits
        dict(name="quantize_gate_nf3", kind="quantize", m=14336, n=4096, r=48, bits=3),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, group):
    """A feature count: mostly multiples of 64 or 128, one in three only a multiple of the pack group."""
    v = _spread(rng, lo, hi)
    step = group if rng.random() < 1 / 3 else max(group, rng.choice((64, 128)))
    return max(step, (v + step // 2) // step * step)


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def draw(rng):
    most = max(_cost(c) for c in listed())
    kind = rng.choice(("forward",) * 6 + ("host", "block", "finetune", "finetune", "qat", "quantize"))
    bits = rng.choice((2, 3, 4, 4))
    # ranks: parameter parity with blocks from 512 down to 16 columns, small ones more often
    r = _spread(rng, 4, 128)
    if kind == "block":
        h = 128 * _spread(rng, 8, 32)
        case = dict(kind=kind, h=h, kv=max(128, h // rng.choice((1, 4, 8)) // 128 * 128), ffn=128 * max(8, round(h * rng.uniform(2.5, 3.5) / 128)),
                    M=_spread(rng, 1, 512), bits=bits, mlp_bits=rng.choice((2, 3, 4)), r=min(r, 64), r_kv=max(2, min(r, 64) // 2),
                    r_mlp=min(64, r + r // 2))
    else:
        m = _width(rng, 256, 14336, 1 if kind in ("forward", "host", "quantize") else GROUP[bits])
        n = _width(rng, 256, 14336, GROUP[bits])
        while m * n > 14336 * 4096:
            if m > n:
                m = m // 2 // GROUP[bits] * GROUP[bits] + m % GROUP[bits]
            else:
                n = n // 2 // GROUP[bits] * GROUP[bits]
        case = dict(kind=kind, m=m, n=n, r=r, bits=bits)
        if kind != "quantize":
            lo, hi = {"forward": (1, 2048), "host": (1, 16), "finetune": (32, 1024), "qat": (32, 1024)}[kind]
            case["M"] = _spread(rng, lo, hi)
    while _cost(case) > most:
        case["M"] //= 2
    return case


# ------------------------------------------------------------------------------------------- inputs
def _book(bits):
    if bits not in _books:
        _books[bits] = inputs.nf_codebook(bits)
    return _books[bits]


def _factors(gen, m, n, r):
    """B and A around the scales that keep S = BA near 0.05 at every rank, all positive."""
    gain = 0.05 * math.sqrt(32.0 / r)
    B = (torch.randn(m, r, generator=gen, device="cuda").abs_() * gain + 0.2 * gain).to(torch.bfloat16)
    A = (torch.randn(r, n, generator=gen, device="cuda").abs_() * gain + 0.2 * gain).to(torch.bfloat16)
    return B, A


def _activations(gen, M, n):
    x = torch.randn(M, n, generator=gen, device="cuda")
    if M >= 256:
        cols = torch.randperm(n, generator=gen, device="cuda")[: max(1, n // 100)]
        x[:, cols] *= 20.0
    return x.to(torch.bfloat16)


def _codes(gen, m, n, bits):
    # uniform codes are uniform bytes in every one of the packed layouts
    return torch.randint(0, 256, (m, n * bits // 8), generator=gen, device="cuda", dtype=torch.uint8)


def _layer(gen, m, n, r, bits):
    B, A = _factors(gen, m, n, r)
    return dict(m=m, n=n, r=r, bits=bits, q=_codes(gen, m, n, bits), B=B, A=A, cb=_book(bits))


def _block_layers(case):
    h, kv, ffn = case["h"], case["kv"], case["ffn"]
    b, mb, r, rk, rm = case["bits"], case["mlp_bits"], case["r"], case["r_kv"], case["r_mlp"]
    return (("q", "attn", h, h, r, b), ("k", "attn", kv, h, rk, b), ("v", "attn", kv, h, rk, b), ("o", "mix", h, h, r, b),
            ("gate", "mlp", ffn, h, rm, mb), ("up", "mlp", ffn, h, rm, mb), ("down", "act", h, ffn, rm, mb))


def prepare(case, seed):
    if not _ready:
        lords.lords_init(torch.cuda.current_device(), 0)
        _ready.append(True)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    st = dict(case)
    if kind == "block":
        h, ffn, M = case["h"], case["ffn"], case["M"]
        xs = {"attn": _activations(gen, M, h), "mix": _activations(gen, M, h), "mlp": _activations(gen, M, h), "act": _activations(gen, M, ffn)}
        st["layers"] = []
        for _, src, m, n, r, bits in _block_layers(case):
            L = _layer(gen, m, n, r, bits)
            L.update(x=xs[src], y=torch.empty(M, m, device="cuda", dtype=torch.bfloat16))
            st["layers"].append(L)
        return st
    m, n, r, bits = case["m"], case["n"], case["r"], case["bits"]
    if kind in ("quantize", "qat"):
        B, A = _factors(gen, m, n, r)
        # weights whose ratio to S spreads over the level range, as weights divided by their block scales do
        W = (torch.randn(m, n, generator=gen, device="cuda") * 0.05).to(torch.bfloat16)
        st.update(W=W, B=B, A=A, cb=_book(bits), q=torch.empty(m, n * bits // 8, device="cuda", dtype=torch.uint8))
    else:
        st.update(_layer(gen, m, n, r, bits))
    if kind == "quantize":
        return st
    M = case["M"]
    x = _activations(gen, M, n)
    if kind == "host":
        st["x"] = x.cpu().pin_memory()
        st["y"] = torch.empty(M, m, dtype=torch.bfloat16, pin_memory=True)
        return st
    st.update(x=x, y=torch.empty(M, m, device="cuda", dtype=torch.bfloat16))
    if kind in ("finetune", "qat"):
        f32 = dict(device="cuda", dtype=torch.float32)
        st.update(dy=torch.randn(M, m, generator=gen, device="cuda").to(torch.bfloat16), qt=torch.empty(n, m * bits // 8, device="cuda", dtype=torch.uint8),
                  dx=torch.empty(M, n, device="cuda", dtype=torch.bfloat16), dB=torch.empty(m, r, **f32), dA=torch.empty(r, n, **f32))
        if kind == "finetune":      # the codes are frozen: their transpose is made once
            lords.lords_transpose_codes(st["q"], bits, m, n, st["qt"])
        else:
            st["dW"] = torch.empty(m, n, **f32)
    return st


# ---------------------------------------------------------------------------------------------- one pass
def run(s):
    kind = s["kind"]
    if kind == "block":
        for L in s["layers"]:
            lords.lords_linear_forward_bits(L["x"], L["q"], L["B"], L["A"], L["cb"], L["bits"], s["M"], L["m"], L["n"], L["r"], L["y"])
        return [L["y"] for L in s["layers"]]
    q, B, A, cb, bits, m, n, r = s["q"], s["B"], s["A"], s["cb"], s["bits"], s["m"], s["n"], s["r"]
    if kind == "quantize":
        lords.lords_quantize_codes(s["W"], B, A, cb, bits, m, n, r, q)
        return q
    M, x, y = s["M"], s["x"], s["y"]
    if kind == "forward":
        lords.lords_linear_forward_bits(x, q, B, A, cb, bits, M, m, n, r, y)
        return y
    if kind == "host":
        lords.lords_linear_forward_host(x, q, B, A, cb, bits, M, m, n, r, y)
        return y
    dy, qt, dx, dB, dA = s["dy"], s["qt"], s["dx"], s["dB"], s["dA"]
    if kind == "qat":               # the weight has moved since the last step: new codes
        lords.lords_quantize_codes(s["W"], B, A, cb, bits, m, n, r, q)
        lords.lords_transpose_codes(q, bits, m, n, qt)
        # the forward kernels may read their weights ahead of the stream's order, so codes that were just
        # written are waited for (include/lords.h)
        torch.cuda.current_stream().synchronize()
    lords.lords_linear_forward_bits(x, q, B, A, cb, bits, M, m, n, r, y)
    lords.lords_linear_backward_input(dy, qt, B, A, cb, bits, M, m, n, r, dx)
    if kind == "finetune":
        lords.lords_linear_backward_factors(dy, x, q, B, A, cb, bits, M, m, n, r, dB, dA)
        return dict(y=y, dx=dx, dB=dB, dA=dA)
    lords.lords_linear_backward_qat(dy, x, s["W"], q, B, A, cb, bits, M, m, n, r, s["dW"], dB, dA)
    return dict(q=q, qt=qt, y=y, dx=dx, dW=s["dW"], dB=dB, dA=dA)


# ------------------------------------------------------------------------------------ floor and tolerance
def work(case):
    kind = case["kind"]
    if kind == "block":
        M, h, ffn = case["M"], case["h"], case["ffn"]
        b, f = 2 * M * (3 * h + ffn), 0            # the four activation tensors
        for _, _, m, n, r, bits in _block_layers(case):
            b += m * n * bits // 8 + 2 * r * (m + n) + 2 * M * m
            f += 2 * M * m * n
        return {"bytes": b, "flops": f}
    m, n, r, bits = case["m"], case["n"], case["r"], case["bits"]
    weights = m * n * bits // 8 + 2 * r * (m + n)
    if kind == "quantize":
        return {"bytes": 2 * m * n + weights, "flops": 2 * m * n * r}
    M = case["M"]
    if kind in ("forward", "host"):
        return {"bytes": weights + 2 * M * (m + n), "flops": 2 * M * m * n}
    # three products over the tokens, and the two folds of dS with the factors; x, dy in, y, dx out
    b = weights + m * n * bits // 8 + 4 * M * (m + n) + 4 * r * (m + n)
    f = 6 * M * m * n + 4 * m * n * r
    if kind == "qat":                              # the weight in, its gradient out, S for codes and quotient
        b += 2 * m * n + 4 * m * n
        f += 2 * m * n * r
    return {"bytes": b, "flops": f}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        # a weight within rounding distance of the midpoint of two levels may get either
        return {"rel": 0.0, "differ": 1e-4}
    # bf16 outputs: half a unit in the last place each (1.7e-3 of the norm), operands rounded once to fp16
    tol = {"rel": 4e-3, "max": 2e-2}
    if kind == "qat":
        tol["differ"] = 1e-4
    return tol
