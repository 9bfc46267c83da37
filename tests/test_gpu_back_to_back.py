"""Calls whose inputs are the outputs of the call before them, with nothing in between (no copy, no synchronisation):
every repetition has other data and writes to the same buffers, so that a value read before the kernel that makes it
has finished would be the one of the repetition before.  Results against the oracle, read after the last repetition."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu

REPS = 6


def buffers(M, N, K, bits, groups):
    return dict(xq=torch.empty((M, K), dtype=torch.int8, device="cuda"), sc=torch.empty(1, device="cuda"),
                rs=torch.empty(M, dtype=torch.int32, device="cuda"),
                packed=torch.empty((N, K * bits // 32), dtype=torch.int32, device="cuda"),
                delta=torch.empty(groups, device="cuda"), q0=torch.empty(groups, device="cuda"))


@pytest.mark.parametrize("V,D,bits,groups,T", [(64, 128, 4, 128, 40), (500, 768, 3, 1, 1200), (3000, 256, 8, 16, 9)])
def test_table_then_lookup(V, D, bits, groups, T):
    ws = qb.workspace(groups=4096)
    rng = np.random.default_rng(V)
    tables = [(rng.standard_normal((V, D)) * 0.02 * (i + 1)).astype(np.float32) for i in range(REPS)]
    ids = [rng.integers(0, V, T).astype(np.int32) for _ in range(REPS)]
    d_tables, d_ids = [gu.dev(t) for t in tables], [gu.dev(i) for i in ids]
    packed = torch.zeros((V, D * bits // 32), dtype=torch.int32, device="cuda")
    outs = [torch.empty((T, D), device="cuda") for _ in range(REPS)]
    torch.cuda.synchronize()
    for i in range(REPS):
        _, delta, q0 = qb.quantize_embedding(d_tables[i], bits, groups, ws, packed=packed)
        qb.embedding_lookup(d_ids[i], packed, delta, q0, D, bits, groups, ws, out=outs[i])
        qb.embedding_lookup(d_ids[i], packed, delta, q0, D, bits, groups, ws, out=outs[i], accumulate=True)
        del delta, q0  # the next repetition's are the same memory
    torch.cuda.synchronize()
    for i in range(REPS):
        _, codes, o_delta, o_q0 = oracle.quantize_embedding(tables[i], bits, groups)
        ref = oracle.embedding_lookup(ids[i], codes, groups, o_delta, o_q0)
        ref = oracle.embedding_lookup(ids[i], codes, groups, o_delta, o_q0, out=ref)
        assert np.array_equal(outs[i].cpu().numpy().view(np.uint32), ref.view(np.uint32)), i
    assert qb.read_status(ws) == qb.QB_OK


# groups in one CTA's registers, a cluster's, the ring, and (a workspace without room for the ring's slots) two passes
@pytest.mark.parametrize("N,K,groups,small_ws", [(128, 256, 8, False), (768, 768, 4, False), (768, 768, 1, False), (768, 768, 1, True)])
@pytest.mark.parametrize("M", (33, 300))
def test_pack_then_gemm_then_requantize(M, N, K, groups, small_ws):
    bits = 4
    ws = qb.workspace(groups=4096)
    if small_ws:
        ws = ws[:512]
    xs = [synth.activations(M, K, seed=i) * np.float32(1 + i) for i in range(REPS)]
    ws_host = [synth.weights(N, K, seed=10 + i) * np.float32(1 + i) for i in range(REPS)]
    d_x, d_w = [gu.dev(x) for x in xs], [gu.dev(w) for w in ws_host]
    b = buffers(M, N, K, bits, groups)
    ys = [torch.empty((M, N), device="cuda") for _ in range(REPS)]
    accs = [torch.empty((M, N), dtype=torch.int32, device="cuda") for _ in range(REPS)]
    again = [None] * REPS
    torch.cuda.synchronize()
    for i in range(REPS):
        qb.quantize_act(d_x[i], ws, b["xq"], b["sc"], b["rs"])
        qb.quantize_pack_weights(d_w[i], bits, groups, ws, packed=b["packed"], delta=b["delta"], q0=b["q0"])
        qb.gemm(b["xq"], b["sc"], b["rs"], b["packed"], b["delta"], b["q0"], None, N, bits, groups, ws, y=ys[i], acc_out=accs[i])
        again[i] = qb.quantize_act(ys[i], ws)
    torch.cuda.synchronize()
    for i in range(REPS):
        _, o_xq, o_s, o_rs = oracle.quantize_act(xs[i])
        _, codes, o_delta, o_q0 = oracle.quantize_weights(ws_host[i], bits, groups)
        o_acc = oracle.int_gemm(o_xq, codes)
        assert np.array_equal(accs[i].cpu().numpy(), o_acc), i
        y = ys[i].cpu().numpy()
        gu.assert_y_close(y, oracle.dequant_epilogue(o_acc, o_rs, o_s, o_delta, o_q0, None, bits, groups))
        _, o_xq, o_s, o_rs = oracle.quantize_act(y)
        assert again[i][1].item() == o_s, i
        assert np.array_equal(again[i][0].cpu().numpy(), o_xq) and np.array_equal(again[i][2].cpu().numpy(), o_rs), i
    assert qb.read_status(ws) == qb.QB_OK


# The quantizer's two launches set up under the GEMM that makes their input (more than 2,368 segments), of one and of several
# segments a row; then under a GEMM that still reads the codes and the row sums which they overwrite.
@pytest.mark.parametrize("M,K,N", [(3001, 768, 768), (1000, 2304, 3072)])
def test_gemm_then_two_launch_quantizer(M, K, N):
    bits, groups = 4, 12
    ws = qb.workspace(groups=64)
    xs = [synth.activations(M, K, seed=i) * np.float32(REPS - i) for i in range(REPS)]  # smaller and smaller
    w = synth.weights(N, K, seed=10)
    d_x, b = [gu.dev(x) for x in xs], buffers(M, N, K, bits, groups)
    qb.quantize_pack_weights(gu.dev(w), bits, groups, ws, packed=b["packed"], delta=b["delta"], q0=b["q0"])
    y = torch.empty((M, N), device="cuda")
    kept, ys = [torch.empty_like(y) for _ in range(REPS)], [torch.empty_like(y) for _ in range(REPS)]
    again = [buffers(M, N, N, bits, groups) for _ in range(REPS)]
    torch.cuda.synchronize()
    for i in range(REPS):
        qb.quantize_act(d_x[i], ws, b["xq"], b["sc"], b["rs"])
        qb.gemm(b["xq"], b["sc"], b["rs"], b["packed"], b["delta"], b["q0"], None, N, bits, groups, ws, y=y)
        qb.quantize_act(y, ws, again[i]["xq"], again[i]["sc"], again[i]["rs"])
        kept[i].copy_(y)
    for i in range(REPS):
        qb.quantize_act(d_x[i], ws, b["xq"], b["sc"], b["rs"])
        qb.gemm(b["xq"], b["sc"], b["rs"], b["packed"], b["delta"], b["q0"], None, N, bits, groups, ws, y=ys[i])
    torch.cuda.synchronize()
    _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, groups)
    sel = gu.sample_rows(M)
    for i in range(REPS):
        _, o_xq, o_s, o_rs = oracle.quantize_act(xs[i])
        gu.assert_y_close(kept[i].cpu().numpy()[sel], oracle.dequant_epilogue(oracle.int_gemm(o_xq[sel], codes), o_rs[sel], o_s, o_delta,
                                                                              o_q0, None, bits, groups))
        assert torch.equal(ys[i], kept[i]), i
        _, o_xq, o_s, o_rs = oracle.quantize_act(kept[i].cpu().numpy())
        assert again[i]["sc"].item() == o_s, i
        assert np.array_equal(again[i]["xq"].cpu().numpy(), o_xq) and np.array_equal(again[i]["rs"].cpu().numpy(), o_rs), i
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("M", (33, 128))
def test_stack_then_batch_quantizer(M):
    bits, groups = 4, 8
    ws = qb.workspace(groups=64)
    shapes = [(768, 768), (3072, 768), (768, 3072)]
    xs = [[synth.activations(M, K, seed=3 * i + j) * np.float32(REPS - i) for j, (_, K) in enumerate(shapes)] for i in range(REPS)]
    w = [synth.weights(N, K, seed=40 + j) for j, (N, K) in enumerate(shapes)]
    b = [buffers(M, N, K, bits, groups) for N, K in shapes]
    for wj, bj in zip(w, b):
        qb.quantize_pack_weights(gu.dev(wj), bits, groups, ws, packed=bj["packed"], delta=bj["delta"], q0=bj["q0"])
    ys = [torch.empty((M, N), device="cuda") for N, _ in shapes]
    kept = [[torch.empty_like(y) for y in ys] for _ in range(REPS)]
    again = [[buffers(M, N, N, bits, groups) for N, _ in shapes] for _ in range(REPS)]
    d_x = [[gu.dev(x) for x in rep] for rep in xs]
    first = [qb.make_act_desc_array([(x, bj["xq"], bj["sc"], bj["rs"]) for x, bj in zip(rep, b)]) for rep in d_x]
    linears = qb.make_desc_array([qb.LinearDesc(bj["xq"], bj["sc"], bj["rs"], bj["packed"], bj["delta"], bj["q0"], None, N, bits, groups, y)
                                  for bj, y, (N, _) in zip(b, ys, shapes)])
    second = [qb.make_act_desc_array([(y, a["xq"], a["sc"], a["rs"]) for y, a in zip(ys, rep)]) for rep in again]
    torch.cuda.synchronize()
    for i in range(REPS):
        qb.quantize_act_batch(first[i], ws)
        qb.layer_linears(linears, ws)
        qb.quantize_act_batch(second[i], ws)
        for k, y in zip(kept[i], ys):
            k.copy_(y)
    torch.cuda.synchronize()
    for j in range(len(shapes)):
        _, codes, o_delta, o_q0 = oracle.quantize_weights(w[j], bits, groups)
        for i in range(REPS):
            _, o_xq, o_s, o_rs = oracle.quantize_act(xs[i][j])
            y = kept[i][j].cpu().numpy()
            gu.assert_y_close(y, oracle.dequant_epilogue(oracle.int_gemm(o_xq, codes), o_rs, o_s, o_delta, o_q0, None, bits, groups))
            _, o_xq, o_s, o_rs = oracle.quantize_act(y)
            a = again[i][j]
            assert a["sc"].item() == o_s, (i, j)
            assert np.array_equal(a["xq"].cpu().numpy(), o_xq) and np.array_equal(a["rs"].cpu().numpy(), o_rs), (i, j)
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("N,K,groups,small_ws", [(128, 256, 8, False), (768, 768, 4, False), (768, 768, 1, False), (768, 768, 1, True)])
def test_fake_quantize_then_pack_then_backward(N, K, groups, small_ws):
    ws = qb.workspace(groups=4096)
    if small_ws:
        ws = ws[:512]
    rng = np.random.default_rng(N)
    hosts = [synth.weights(N, K, seed=20 + i) * np.float32(1 + i) for i in range(REPS)]
    grads = [rng.standard_normal((N, K)).astype(np.float32) for _ in range(REPS)]
    d_w, d_g = [gu.dev(w) for w in hosts], [gu.dev(g) for g in grads]
    lo, hi = gu.dev(np.full(groups, -0.02, np.float32)), gu.dev(np.full(groups, 0.02, np.float32))
    wq = torch.empty((N, K), device="cuda")
    kept, packs, backs = [torch.empty((N, K), device="cuda") for _ in range(REPS)], [None] * REPS, [None] * REPS
    torch.cuda.synchronize()
    for i in range(REPS):
        qb.fake_quantize_weights(d_w[i], 4, groups, ws, wq=wq)
        packs[i] = qb.quantize_pack_weights(wq, 4, groups, ws)
        qb.fake_quantize_weights(wq, 8, groups, ws, wq=kept[i])
        backs[i] = qb.ste_backward(d_g[i], kept[i], groups, lo, hi)
    torch.cuda.synchronize()
    for i in range(REPS):
        o_wq = oracle.fake_quantize_weights(hosts[i], 4, groups)[1]
        _, codes, o_delta, o_q0 = oracle.quantize_weights(o_wq, 4, groups)
        assert np.array_equal(gu.words_np(packs[i][0]), oracle.pack(codes, 4)), i
        assert np.array_equal(packs[i][1].cpu().numpy(), o_delta) and np.array_equal(packs[i][2].cpu().numpy(), o_q0)
        o_kept = oracle.fake_quantize_weights(o_wq, 8, groups)[1]
        assert np.array_equal(kept[i].cpu().numpy(), o_kept), i
        assert np.array_equal(backs[i].cpu().numpy(), oracle.ste_backward(grads[i], o_kept, groups, lo.cpu().numpy(), hi.cpu().numpy())), i
    assert qb.read_status(ws) == qb.QB_OK
