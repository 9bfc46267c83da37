"""Calls on a stream that has a part of the device's SMs (a green context): the kernels whose blocks must all be resident
give way to the forms that need no residency, with the same results."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def part():
    contexts = pytest.importorskip("torch.cuda.green_contexts")
    if not contexts.SUPPORTED:
        pytest.skip("torch without green contexts")
    torch.zeros(1, device="cuda")
    return contexts.GreenContext.create(16, 0)


def in_part(part, call):
    torch.cuda.synchronize()
    part.set_context()
    try:
        call()
        torch.cuda.synchronize()
    finally:
        part.pop_context()


# on the whole device: one cluster of one and of 8 CTAs; 5 clusters; 152 CTAs of 16 warps, more than 16 SMs hold; two launches
@pytest.mark.parametrize("M,K", [(3, 256), (256, 1024), (320, 1024), (2368, 1024), (6000, 768)])
def test_quantize_act(part, M, K):
    ws = qb.workspace(groups=64)
    for seed in (1, 2):
        x = synth.activations(M, K, seed=seed) * np.float32(1.0 / seed)
        xd = gu.dev(x)
        xq, sc, rs = (gu.poison(torch.empty(s, dtype=t, device="cuda"))
                      for s, t in (((M, K), torch.int8), (1, torch.float32), (M, torch.int32)))
        in_part(part, lambda: qb.quantize_act(xd, ws, xq, sc, rs))
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s
        assert np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
        whole = qb.quantize_act(xd, ws)  # and on the whole device, with the workspace that the call above left
        assert torch.equal(whole[0], xq) and torch.equal(whole[2], rs)
    assert qb.read_status(ws) == qb.QB_OK


# a CTA's registers, a cluster's, and the ring (one range per matrix), which takes every SM
@pytest.mark.parametrize("groups", (768, 4, 1))
def test_quantize_weights(part, groups):
    ws = qb.workspace(groups=4096)
    w = synth.weights(768, 768, seed=groups)
    wd = gu.dev(w)
    packed = torch.full((768, 768 * 3 // 32), -1, dtype=torch.int32, device="cuda")
    delta, q0 = torch.empty(groups, device="cuda"), torch.empty(groups, device="cuda")
    wq = torch.empty((768, 768), device="cuda")
    in_part(part, lambda: qb.quantize_pack_weights(wd, 3, groups, ws, packed=packed, delta=delta, q0=q0))
    in_part(part, lambda: qb.fake_quantize_weights(wd, 4, groups, ws, wq=wq))
    _, codes, o_delta, o_q0 = oracle.quantize_weights(w, 3, groups)
    assert np.array_equal(gu.words_np(packed), oracle.pack(codes, 3))
    assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
    o_wq = oracle.fake_quantize_weights(w, 4, groups)[1]
    assert np.array_equal(wq.cpu().numpy().view(np.uint32), o_wq.view(np.uint32))
    whole = qb.quantize_pack_weights(wd, 3, groups, ws)
    assert torch.equal(whole[0], packed)
    assert qb.read_status(ws) == qb.QB_OK


# Under capture nothing refuses a cooperative launch that does not fit: the graph would wait for room for ever.
@pytest.mark.parametrize("what", ("one cluster", "several clusters", "two launches", "registers", "clusters", "ring"))
def test_captured(part, what):
    ws = qb.workspace(groups=4096)
    stream = torch.cuda.ExternalStream(part.Stream().cuda_stream)
    if what in ("registers", "clusters", "ring"):
        groups = {"registers": 768, "clusters": 4, "ring": 1}[what]
        w = gu.dev(synth.weights(768, 768, seed=groups))
        outs = list(qb.quantize_pack_weights(w, 3, groups, ws))
        outs.append(qb.fake_quantize_weights(w, 4, groups, ws)[0])

        def call():
            qb.quantize_pack_weights(w, 3, groups, ws, packed=outs[0], delta=outs[1], q0=outs[2])
            qb.fake_quantize_weights(w, 4, groups, ws, wq=outs[3])
    else:
        M = {"one cluster": 256, "several clusters": 2368, "two launches": 6000}[what]
        x = gu.dev(synth.activations(M, 768, seed=M))
        outs = list(qb.quantize_act(x, ws))

        def call():
            qb.quantize_act(x, ws, *outs)

    expected = [o.clone() for o in outs]  # the whole device's, which the other tests compare with the oracle
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        g.capture_begin()
        try:
            call()
        finally:
            g.capture_end()
        for _ in range(2):
            for o in outs:
                gu.poison(o)
            g.replay()
            stream.synchronize()  # (synchronising the device does not wait for a green context's stream)
            assert all(torch.equal(a, b) for a, b in zip(outs, expected))
            stream.synchronize()
    assert qb.read_status(ws) == qb.QB_OK
