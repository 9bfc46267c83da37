"""The quantizers under stream capture, in every form that they launch: replays read the buffers as they are then, and
calls outside the graph share its workspace."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


def captured(call):
    call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


# one cluster, several clusters (cooperative) of 8 and of 16 warps a CTA, two launches
@pytest.mark.parametrize("M,K", [(64, 768), (320, 1024), (2368, 256), (6000, 768)])
def test_quantize_act(M, K):
    ws = qb.workspace(groups=64)
    x = gu.dev(synth.activations(M, K, seed=1) * np.float32(9.0))
    xq, sc, rs = qb.quantize_act(x, ws)
    g = captured(lambda: qb.quantize_act(x, ws, xq, sc, rs))
    for seed in (2, 3, 4):
        host = synth.activations(M, K, seed=seed) * np.float32(1.0 / seed)
        x.copy_(torch.from_numpy(host))
        other = qb.quantize_act(gu.dev(host), ws)  # between replays, on the same workspace
        g.replay()
        _, o_xq, o_s, o_rs = oracle.quantize_act(host)
        for q, s, r in ((xq, sc, rs), other):
            assert s.item() == o_s
            assert np.array_equal(q.cpu().numpy(), o_xq) and np.array_equal(r.cpu().numpy(), o_rs)
    assert qb.read_status(ws) == qb.QB_OK


# a CTA's registers, a cluster's, the ring (cooperative), and two passes in a workspace without room for its slots
@pytest.mark.parametrize("groups,small_ws", [(64, False), (4, False), (1, False), (1, True)])
def test_quantize_weights(groups, small_ws):
    ws = qb.workspace(groups=4096)
    if small_ws:
        ws = ws[:512]
    w = gu.dev(synth.weights(768, 768, seed=1) * np.float32(9.0))
    packed, delta, q0 = qb.quantize_pack_weights(w, 3, groups, ws)
    wq = torch.empty_like(w)

    def call():
        qb.quantize_pack_weights(w, 3, groups, ws, packed=packed, delta=delta, q0=q0)
        qb.fake_quantize_weights(w, 4, groups, ws, wq=wq)

    g = captured(call)
    for seed in (2, 3, 4):
        host = synth.weights(768, 768, seed=seed) * np.float32(1.0 / seed)
        w.copy_(torch.from_numpy(host))
        g.replay()
        _, codes, o_delta, o_q0 = oracle.quantize_weights(host, 3, groups)
        assert np.array_equal(gu.words_np(packed), oracle.pack(codes, 3))
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
        o_wq = oracle.fake_quantize_weights(host, 4, groups)[1]
        assert np.array_equal(wq.cpu().numpy().view(np.uint32), o_wq.view(np.uint32))
    assert qb.read_status(ws) == qb.QB_OK


def test_embedding():
    ws = qb.workspace(groups=4096)
    rng = np.random.default_rng(5)
    table = torch.rand((600, 256), device="cuda")
    ids = torch.zeros(900, dtype=torch.int32, device="cuda")
    packed = torch.empty((600, 256 * 4 // 32), dtype=torch.int32, device="cuda")
    out = torch.empty((900, 256), device="cuda")

    def call():
        _, delta, q0 = qb.quantize_embedding(table, 4, 16, ws, packed=packed)
        qb.embedding_lookup(ids, packed, delta, q0, 256, 4, 16, ws, out=out)
        qb.embedding_lookup(ids, packed, delta, q0, 256, 4, 16, ws, out=out, accumulate=True)

    g = captured(call)
    for seed in range(3):
        e = (rng.standard_normal((600, 256)) * 0.02 * (3 - seed)).astype(np.float32)
        i = rng.integers(0, 600, 900).astype(np.int32)
        table.copy_(torch.from_numpy(e))
        ids.copy_(torch.from_numpy(i))
        g.replay()
        _, codes, o_delta, o_q0 = oracle.quantize_embedding(e, 4, 16)
        ref = oracle.embedding_lookup(i, codes, 16, o_delta, o_q0)
        ref = oracle.embedding_lookup(i, codes, 16, o_delta, o_q0, out=ref)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    assert qb.read_status(ws) == qb.QB_OK
