"""The work that users of libqbert have it do, as cases for timing and for comparing results.

A case is a dict of plain values; ``kind`` names the job:

* ``linear``        one quantized linear on a fresh activation tensor: ``quantize_act`` then ``gemm`` /
                    ``gemm_bf16`` (weights were packed when the model was loaded);
* ``stack``         the linears of one or more encoder layers: ``quantize_act_batch`` then
                    ``layer_linears`` / ``layer_linears_bf16``;
* ``ffn_chain``     a feed-forward block that stays at 8 bits inside: ``quantize_act``, ``gemm_i8`` on a
                    calibrated scale, ``rowsum_i8``, ``gemm``;
* ``pack``          loading a model: ``quantize_pack_weights_batch`` over its fp32 matrices;
* ``finetune``      the quantizer's part of a fine-tuning step: ``fake_quantize_weights_batch`` forward, one
                    ``ste_backward`` per matrix;
* ``embed_pack``    quantizing an embedding table;
* ``embed_lookup``  word plus position embedding of a batch of tokens.

Inputs have the distributions of ``paper_1909_05840_b200.synth`` (normal activations with two outlier
channels, normal weights with 1 % Laplace outliers), drawn on the GPU.
"""
import math

import torch

import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

MIXED = "mixed"  # per-layer widths as the mixed-precision assignment gives them (half of the layers 2 bits)


def listed():
    return [
        # The pooler of a small batch: one token of each of 32 sequences through a square 8-bit linear.  The
        # smallest call: latency and launches.
        {"name": "pooler_m32_8bit", "kind": "linear", "M": 32, "N": 768, "K": 768, "bits": 8, "groups": 128, "out": "fp32"},
        # The query projection of 8 sequences of 128 tokens, one range per attention head.
        {"name": "query_m1024_4bit", "kind": "linear", "M": 1024, "N": 768, "K": 768, "bits": 4, "groups": 12, "out": "fp32"},
        # Serving one sequence of 128 tokens through all twelve layers of a mixed-precision model: 48 linears.
        {"name": "stack12_m128_mixed", "kind": "stack", "M": 128, "hidden": 768, "ffn": 3072, "layers": 12, "bits": MIXED, "groups": 128, "out": "fp32"},
        # One encoder layer at batch 32 x 128 tokens, 3 bits.
        {"name": "layer_m4096_3bit", "kind": "stack", "M": 4096, "hidden": 768, "ffn": 3072, "layers": 1, "bits": "3", "groups": 128, "out": "fp32"},
        # Two layers of the large encoder at batch 64 x 384 tokens, 4 bits: throughput.
        {"name": "large_m24576_4bit", "kind": "stack", "M": 24576, "hidden": 1024, "ffn": 4096, "layers": 2, "bits": "4", "groups": 128, "out": "fp32"},
        # A ragged batch (padding removed: an odd number of tokens) through a layer of the large encoder,
        # 2 bits, outputs handed on as bfloat16.
        {"name": "large_m5003_2bit_bf16", "kind": "stack", "M": 5003, "hidden": 1024, "ffn": 4096, "layers": 1, "bits": "2", "groups": 128, "out": "bf16"},
        # A feed-forward block whose inner activations stay int8, 16 sequences of 384 tokens.
        {"name": "ffn_chain_m6144_4bit", "kind": "ffn_chain", "M": 6144, "hidden": 1024, "ffn": 4096, "bits": 4, "groups": 128},
        # Loading a mixed-precision base model: 48 matrices, 128 groups per attention matrix.
        {"name": "pack_base_mixed_g128", "kind": "pack", "hidden": 768, "ffn": 3072, "layers": 12, "bits": MIXED, "groups": 128},
        # The same model at one range per matrix (layer-wise quantization), 4 bits.
        {"name": "pack_base_4bit_g1", "kind": "pack", "hidden": 768, "ffn": 3072, "layers": 12, "bits": "4", "groups": 1},
        # A quantization-aware fine-tuning step over four layers with clipped ranges.
        {"name": "finetune_base_4bit", "kind": "finetune", "hidden": 768, "ffn": 3072, "layers": 4, "bits": "4", "groups": 128},
        # Quantizing the word embedding table (4 bits, 128 groups of columns).
        {"name": "embed_pack_30522_4bit", "kind": "embed_pack", "V": 30522, "D": 768, "bits": 4, "groups": 128},
        # Embedding a batch of 64 x 384 tokens: 4-bit word table, then the 8-bit position table added.
        {"name": "embed_lookup_24576", "kind": "embed_lookup", "T": 24576, "V": 30522, "P": 512, "D": 768, "bits": 4, "groups": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _divisor(rng, n, most=768):
    return rng.choice([d for d in range(1, min(n, most) + 1) if n % d == 0])


def draw(rng):
    """One more case of the same ranges: batch sizes over their logarithm and mostly odd, hidden sizes in steps of
    128 up to the large encoder's, every bit width, from one range per matrix to one per row."""
    kind = rng.choice(["linear", "linear", "stack", "stack", "ffn_chain", "pack", "finetune", "embed_pack", "embed_lookup"])
    hidden = 128 * rng.randint(2, 8)
    ffn = 4 * hidden
    bits = rng.choice(synth.BITS_CHOICES)
    groups = _divisor(rng, hidden)
    out = rng.choice(["fp32", "fp32", "bf16"])
    if kind == "linear":
        # output features of any number (a task head may have 9), input features in steps of 128
        N = _log_int(rng, 8, 4096)
        N = N if rng.random() < 0.5 else max(64, N // 64 * 64)
        return {"kind": kind, "M": _log_int(rng, 1, 8192), "N": N, "K": 128 * rng.randint(1, 32), "bits": bits,
                "groups": _divisor(rng, N), "out": out}
    if kind == "stack":
        # the product of tokens and layers stays within the largest listed stack
        M = _log_int(rng, 16, 24576)
        layers = min(rng.randint(1, 12), max(1, 2 * 24576 // M))
        return {"kind": kind, "M": M, "hidden": hidden, "ffn": ffn, "layers": layers,
                "bits": rng.choice([MIXED, str(bits)]), "groups": groups, "out": out}
    if kind == "ffn_chain":
        return {"kind": kind, "M": _log_int(rng, 64, 12288), "hidden": hidden, "ffn": ffn, "bits": bits, "groups": groups}
    if kind == "pack":
        return {"kind": kind, "hidden": hidden, "ffn": ffn, "layers": rng.randint(1, 12),
                "bits": rng.choice([MIXED, str(bits)]), "groups": groups}
    if kind == "finetune":
        return {"kind": kind, "hidden": hidden, "ffn": ffn, "layers": rng.randint(1, 6), "bits": str(bits), "groups": groups}
    if kind == "embed_pack":
        return {"kind": kind, "V": _log_int(rng, 512, 65536), "D": hidden, "bits": bits, "groups": groups}
    return {"kind": kind, "T": _log_int(rng, 16, 49152), "V": _log_int(rng, 2048, 65536), "P": 512, "D": hidden,
            "bits": bits, "groups": groups}


# ---- inputs ------------------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _activations(g, M, K):
    x = torch.randn((M, K), generator=g, device="cuda")
    cols = torch.randperm(K, generator=g, device="cuda")[:2]
    x[:, cols] *= 20.0
    return x


def _weights(g, N, K):
    w = torch.randn((N, K), generator=g, device="cuda").mul_(0.02)
    u = torch.rand((N, K), generator=g, device="cuda")
    # one element in a hundred is a Laplace draw, by inversion of what is left of u
    t = u * 100.0 - 0.5
    laplace = -0.1 * torch.sign(t) * torch.log1p(-2.0 * t.abs().clamp(max=0.4999999))
    return torch.where(u < 0.01, laplace, w)


def _bias(g, N):
    return torch.randn(N, generator=g, device="cuda").mul_(0.02)


def _layer_bits(case):
    if case["bits"] == MIXED:
        return synth.mixed_bits(case["layers"], synth.seed_for(2))
    return (int(case["bits"]),) * case["layers"]


def _linears(case):
    """(shape, bits) of every linear of the case's layers, in execution order."""
    shapes = synth.encoder_linears(case["hidden"], case["ffn"], case["groups"])
    return [(s, b) for b in _layer_bits(case) for s in shapes]


class _Arena:
    """One buffer cut into the tensors of a stack, each at a 256-byte boundary."""

    def __init__(self, shapes, dtype):
        size = torch.empty((), dtype=dtype).element_size()
        self.begin, total = [], 0
        for s in shapes:
            self.begin.append(total)
            total += -(-math.prod(s) * size // 256) * 256 // size
        self.flat = torch.zeros(total, dtype=dtype, device="cuda")
        self.parts = [self.flat[b:b + math.prod(s)].view(s) for b, s in zip(self.begin, shapes)]


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "linear":
        st["ws"] = qb.workspace(groups=case["groups"])
        st["x"] = _activations(g, case["M"], case["K"])
        st["weight"] = qb.quantize_pack_weights(_weights(g, case["N"], case["K"]), case["bits"], case["groups"], st["ws"])
        st["bias"] = _bias(g, case["N"])
    elif kind == "stack":
        lin = _linears(case)
        M = case["M"]
        st["ws"] = qb.workspace(groups=max(64, max(s.groups for s, _ in lin)))
        ys = _Arena([(M, s.N) for s, _ in lin], torch.bfloat16 if case["out"] == "bf16" else torch.float32)
        xqs = _Arena([(M, s.K) for s, _ in lin], torch.int8)
        scales = torch.zeros(len(lin), device="cuda")
        rowsums = torch.zeros((len(lin), M), dtype=torch.int32, device="cuda")
        acts, descs, keep = [], [], []
        for i, (s, b) in enumerate(lin):
            x = _activations(g, M, s.K)
            w = qb.quantize_pack_weights(_weights(g, s.N, s.K), b, s.groups, st["ws"])
            bias = _bias(g, s.N)
            keep.append((x, w, bias))
            acts.append((x, xqs.parts[i], scales[i:i + 1], rowsums[i]))
            descs.append(qb.LinearDesc(xqs.parts[i], scales[i:i + 1], rowsums[i], *w, bias, s.N, b, s.groups, ys.parts[i]))
        st["acts"] = qb.make_act_desc_array(acts)
        st["descs"] = qb.make_desc_array(descs)
        st["keep"] = keep
        st["outputs"] = [ys.flat, xqs.flat, scales, rowsums]
    elif kind == "ffn_chain":
        M, H, F, b, G = case["M"], case["hidden"], case["ffn"], case["bits"], case["groups"]
        st["ws"] = qb.workspace(groups=G)
        st["x"] = _activations(g, M, H)
        st["up"] = qb.quantize_pack_weights(_weights(g, F, H), b, G, st["ws"])
        st["down"] = qb.quantize_pack_weights(_weights(g, H, F), b, G, st["ws"])
        st["bias_up"], st["bias_down"] = _bias(g, F), _bias(g, H)
        # the static scale of the inner activations, calibrated on a few rows
        act = qb.quantize_act(st["x"][:256].contiguous(), st["ws"])
        y = qb.gemm(*act, *st["up"], st["bias_up"], F, b, G, st["ws"])
        st["inner_scale"] = (y.abs().max() / 127.0).reshape(1)
    elif kind == "pack":
        lin = _linears(case)
        words = _Arena([(s.N, s.K * b // 32) for s, b in lin], torch.int32)
        deltas = _Arena([(s.groups,) for s, _ in lin], torch.float32)
        q0s = _Arena([(s.groups,) for s, _ in lin], torch.float32)
        ws_ = [_weights(g, s.N, s.K) for s, _ in lin]
        st["descs"] = qb.make_weight_desc_array([(w, b, s.groups, p, d, z) for w, (s, b), p, d, z in
                                                 zip(ws_, lin, words.parts, deltas.parts, q0s.parts)])
        st["keep"] = ws_
        st["outputs"] = [words.flat, deltas.flat, q0s.flat]
        st["ws"] = qb.workspace(groups=max(32, sum(s.groups for s, _ in lin)))
    elif kind == "finetune":
        lin = _linears(case)
        wqs = _Arena([(s.N, s.K) for s, _ in lin], torch.float32)
        grads = _Arena([(s.N, s.K) for s, _ in lin], torch.float32)
        deltas = _Arena([(s.groups,) for s, _ in lin], torch.float32)
        q0s = _Arena([(s.groups,) for s, _ in lin], torch.float32)
        items, back = [], []
        for i, (s, b) in enumerate(lin):
            w = _weights(g, s.N, s.K)
            gq = torch.randn((s.N, s.K), generator=g, device="cuda").mul_(1e-3)
            lo = torch.rand(s.groups, generator=g, device="cuda").mul_(0.05).sub_(0.15)
            hi = torch.rand(s.groups, generator=g, device="cuda").mul_(0.05).add_(0.10)
            items.append((w, b, s.groups, wqs.parts[i], deltas.parts[i], q0s.parts[i]))
            back.append((gq, w, s.groups, lo, hi, grads.parts[i]))
        st["descs"] = qb.make_weight_desc_array(items)
        for d, (_, _, _, lo, hi, _) in zip(st["descs"], back):
            d.range_lo, d.range_hi = lo.data_ptr(), hi.data_ptr()
        st["back"] = back
        st["outputs"] = [wqs.flat, deltas.flat, q0s.flat, grads.flat]
        st["ws"] = qb.workspace(groups=max(32, sum(s.groups for s, _ in lin)))
    elif kind == "embed_pack":
        st["table"] = _weights(g, case["V"], case["D"])
        st["ws"] = qb.workspace(groups=case["D"])
    elif kind == "embed_lookup":
        D, G, T = case["D"], case["groups"], case["T"]
        st["ws"] = qb.workspace(groups=D)
        st["word"] = qb.quantize_embedding(_weights(g, case["V"], D), case["bits"], G, st["ws"])
        st["position"] = qb.quantize_embedding(_weights(g, case["P"], D), 8, G, st["ws"])
        # token frequencies fall off as in text: a few ids make up most of the batch
        u = torch.rand(T, generator=g, device="cuda")
        st["ids"] = (torch.exp(u * math.log(case["V"])).long().clamp(max=case["V"]) - 1).to(torch.int32)
        st["positions"] = (torch.arange(T, device="cuda") % min(384, case["P"])).to(torch.int32)
    else:
        raise ValueError(f"unknown kind {kind!r}")
    return st


def run(st):
    c = st["case"]
    kind, ws = c["kind"], st["ws"]
    if kind == "linear":
        act = qb.quantize_act(st["x"], ws)
        gemm = qb.gemm_bf16 if c["out"] == "bf16" else qb.gemm
        return [gemm(*act, *st["weight"], st["bias"], c["N"], c["bits"], c["groups"], ws), *act]
    if kind == "stack":
        qb.quantize_act_batch(st["acts"], ws)
        (qb.layer_linears_bf16 if c["out"] == "bf16" else qb.layer_linears)(st["descs"], ws)
        return st["outputs"]
    if kind == "ffn_chain":
        act = qb.quantize_act(st["x"], ws)
        inner = qb.gemm_i8(*act, *st["up"], st["bias_up"], c["ffn"], c["bits"], c["groups"], st["inner_scale"], ws)
        sums = qb.rowsum_i8(inner)
        y = qb.gemm(inner, st["inner_scale"], sums, *st["down"], st["bias_down"], c["hidden"], c["bits"], c["groups"], ws)
        return [y, inner, sums]
    if kind == "pack":
        qb.quantize_pack_weights_batch(st["descs"], ws)
        return st["outputs"]
    if kind == "finetune":
        qb.fake_quantize_weights_batch(st["descs"], ws)
        for grad_q, w, groups, lo, hi, grad_w in st["back"]:
            qb.ste_backward(grad_q, w, groups, lo, hi, grad_w)
        return st["outputs"]
    if kind == "embed_pack":
        return list(qb.quantize_embedding(st["table"], c["bits"], c["groups"], ws))
    out = qb.embedding_lookup(st["ids"], *st["word"], c["D"], c["bits"], c["groups"], ws)
    return qb.embedding_lookup(st["positions"], *st["position"], c["D"], 8, c["groups"], ws, out=out, accumulate=True)


def work(case):
    kind = case["kind"]
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        y = 2 if case["out"] == "bf16" else 4
        return {"bytes": 5 * M * K + 4 * M + N * K * case["bits"] / 8 + y * M * N + 4 * N + 8 * case["groups"],
                "flops": 2 * M * N * K}
    if kind == "stack":
        M, y = case["M"], 2 if case["out"] == "bf16" else 4
        lin = _linears(case)
        return {"bytes": sum(5 * M * s.K + 4 * M + s.N * s.K * b / 8 + y * M * s.N + 4 * s.N + 8 * s.groups for s, b in lin),
                "flops": sum(2 * M * s.N * s.K for s, _ in lin)}
    if kind == "ffn_chain":
        M, H, F = case["M"], case["hidden"], case["ffn"]
        return {"bytes": 5 * M * H + M * F + 8 * M + 2 * H * F * case["bits"] / 8 + 4 * M * H + 4 * (H + F),
                "flops": 4 * M * H * F}
    if kind == "pack":
        return {"bytes": sum(s.N * s.K * (4 + b / 8) + 8 * s.groups for s, b in _linears(case)), "flops": 0}
    if kind == "finetune":
        return {"bytes": sum(s.N * s.K * 20 + 24 * s.groups for s, _ in _linears(case)), "flops": 0}
    if kind == "embed_pack":
        return {"bytes": case["V"] * case["D"] * (4 + case["bits"] / 8) + 8 * case["groups"], "flops": 0}
    # every looked-up row of codes once, the table's rows no more than once each, the sum written once
    T, D = case["T"], case["D"]
    return {"bytes": D * (min(T, case["V"]) * case["bits"] / 8 + min(T, case["P"]) + 4 * T) + 8 * T, "flops": 0}


def tolerance(case):
    """Codes, packed words, steps and integer sums are exact.  The dequantized fp32 values are two fused
    multiply-adds on exact integers: against the same sum in 64 bits 1.3e-7 (largest 2.5e-6 where the terms
    cancel), measured at K = 1024.  Rounded to bfloat16, the few values that then fall on the other side of a
    tie move by one part in 128 (2.3e-5 in all), and a re-quantized value by one code (below 5e-6 of them).
    Stated: about four times that."""
    kind = case["kind"]
    if kind in ("pack", "embed_pack"):
        return "exact"
    if kind == "ffn_chain":
        return {"rel": 2e-4, "max": 4e-3, "differ": 1e-5}
    if case.get("out") == "bf16":
        return {"rel": 1e-4, "max": 8e-3, "differ": 0.0}
    return {"rel": 5e-7, "max": 1e-5, "differ": 0.0}
