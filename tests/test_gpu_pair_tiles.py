"""CTA pairs with 192-token tiles: chosen when 256-token tiles would leave the pairs of SMs idle in the last round.
Ragged tokens and neurons, one K block to 32 (the ring has five stages; from nine on the token tiles are fetched ahead into
L2), every width and output type; single linears, and stacks whose linears differ in K."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


# 1.1 to 1.3 rounds of 256-token tiles over 74 pairs; and 1.6 rounds, which 256-token tiles serve
@pytest.mark.parametrize("bits", (2, 3, 4, 8))
@pytest.mark.parametrize("M,N,K,tokens", [(6100, 1000, 256, 192), (6100, 1000, 1152, 192), (5000, 1024, 128, 192), (2048, 3000, 768, 192),
                                          (5003, 1000, 4096, 192), (6144, 1040, 1152, 256)])
def test_pairs_with_192_token_tiles(bits, M, N, K, tokens):
    ws = qb.workspace(groups=64)
    shape = (qb.LinearDescC * 1)(qb.LinearDescC(M=M, N=N, K=K, bits=bits))
    assert all(qb.layer_linears_tile_tokens(shape, out) == tokens for out in (torch.float32, torch.bfloat16, torch.int8))
    x, w, b = synth.activations(M, K, seed=M + bits), synth.weights(N, K, seed=N), synth.bias(N, seed=K)
    r = gu.check_linear(x, w, b, bits, 8, ws, rows=gu.sample_rows(M, tile=192, per_tile=2, seed=K), use_omp=True)
    args = (r["xq"], r["act_scale"], r["rowsum"], r["packed"], r["delta"], r["q0"], gu.dev(b), N, bits, 8)
    y = r["y"]
    # the narrow outputs are roundings of the fp32 value
    assert torch.equal(qb.gemm_bf16(*args, ws), y.bfloat16())
    step = (y.abs().max() / 100.0).reshape(1)
    yq = qb.gemm_i8(*args, step, ws)
    assert torch.equal(yq, torch.round(y * (torch.ones_like(step) / step)).clamp(-127, 127).to(torch.int8))
    assert qb.read_status(ws) == qb.QB_OK


# tiles of unequal length, dealt from the list of loads: few tokens (one or two token tiles a linear), ragged neurons
@pytest.mark.parametrize("bits", (2, 3, 4, 8))
@pytest.mark.parametrize("M", (131, 192, 300, 384))
def test_stacks_with_192_token_tiles(bits, M):
    ws = qb.workspace(groups=64)
    shapes = [(2300, 384), (776, 768), (3080, 128), (1000, 1152), (2048, 2048), (4, 640)] * 2
    lins, descs = [], []
    for i, (N, K) in enumerate(shapes):
        x, w, b = synth.activations(M, K, seed=i), synth.weights(N, K, seed=i + 50), synth.bias(N, seed=i)
        act, pack = qb.quantize_act(gu.dev(x), ws), qb.quantize_pack_weights(gu.dev(w), bits, 4, ws)
        y = gu.poison(torch.empty((M, N), dtype=torch.float32, device="cuda"))
        lins.append((x, w, b))
        descs.append(qb.LinearDesc(*act, *pack, gu.dev(b), N, bits, 4, y))
    assert qb.layer_linears_launch_count(descs) == 1
    assert all(qb.layer_linears_tile_tokens(descs, out) == 192 for out in (torch.float32, torch.bfloat16, torch.int8))
    qb.layer_linears(descs, ws)
    for (x, w, b), d in list(zip(lins, descs))[: len(shapes) // 2]:  # (the second half: the same shapes, other data)
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, 4)
        rows = gu.sample_rows(M, tile=192, per_tile=4, seed=M)
        o_acc = oracle.int_gemm(o_xq[rows], codes, omp=True)
        gu.assert_y_close(d.y.cpu().numpy()[rows], oracle.dequant_epilogue(o_acc, o_rs[rows], o_s, o_delta, o_q0, b, bits, 4))
    for d in descs:  # all of it, as single linears give it (other tiles, other kernels)
        single = qb.gemm(d.xq, d.act_scale, d.rowsum, d.packed, d.delta, d.q0, d.bias, d.N, bits, 4, ws)
        assert torch.equal(single, d.y)
    fp32 = [d.y for d in descs]
    for d in descs:
        d.y = gu.poison(torch.empty((M, d.N), dtype=torch.bfloat16, device="cuda"))
    qb.layer_linears_bf16(descs, ws)
    assert all(torch.equal(d.y, y.bfloat16()) for d, y in zip(descs, fp32))
    steps = [(y.abs().max() / 100.0).reshape(1) for y in fp32]
    for d in descs:
        d.y = gu.poison(torch.empty((M, d.N), dtype=torch.int8, device="cuda"))
    qb.layer_linears_i8(descs, steps, ws)
    for d, y, step in zip(descs, fp32, steps):
        assert torch.equal(d.y, torch.round(y * (torch.ones_like(step) / step)).clamp(-127, 127).to(torch.int8))
    assert qb.read_status(ws) == qb.QB_OK
