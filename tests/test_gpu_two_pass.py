"""The weight quantizer's two passes, against the oracle: they serve groups beyond a cluster's registers where the
workspace has no room for the ring's slots (8 bytes a group are enough), and groups of more than 27 MB; the ring serves the
same shapes with the workspace that qb_workspace_bytes asks for, with the same results."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


def small(ws, groups):
    n = (256 + 8 * groups + 255) // 256 * 256
    assert n < 256 + 160 * 8 * groups
    return ws[:n]


# units per group: 4,608; 2,368 with a group boundary inside a row of the launch; 4,096 = rows of 512; 2,305; ragged
SHAPES = [(768, 768, 1), (74, 8192, 2), (8, 65536, 1), (2305, 128, 1), (999, 1152, 3)]


@pytest.mark.parametrize("bits", (2, 3, 4, 8))
@pytest.mark.parametrize("N,K,groups", SHAPES)
def test_single_matrices(N, K, groups, bits):
    ws = qb.workspace(groups=64)
    for seed in (1, 2):  # the second has smaller ranges: tables that were not cleared would show
        w = synth.weights(N, K, seed=seed) * np.float32(1.0 / seed)
        packed, delta, q0 = gu.gpu_quantize_weights(w, bits, groups, small(ws, groups))
        _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, groups, omp=True)
        assert np.array_equal(gu.words_np(packed), oracle.pack(codes, bits))
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
        wq, d, z = qb.fake_quantize_weights(gu.dev(w), bits, groups, small(ws, groups))
        o_wq = oracle.fake_quantize_weights(w, bits, groups, omp=True)[1]
        assert np.array_equal(wq.cpu().numpy().view(np.uint32), o_wq.view(np.uint32))
        assert torch.equal(d, delta) and torch.equal(z, q0)
        ring = qb.quantize_pack_weights(gu.dev(w), bits, groups, ws)
        assert torch.equal(ring[0], packed) and torch.equal(ring[1], delta) and torch.equal(ring[2], q0)
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("fake", (False, True))
def test_batch(fake):
    ws = qb.workspace(groups=64)
    items, host = [], []
    for i, (N, K, G) in enumerate(SHAPES + [(768, 768, 4)]):
        w = synth.weights(N, K, seed=30 + i)
        bits = (2, 3, 4, 8)[i % 4]
        out = torch.empty((N, K), device="cuda") if fake else torch.empty((N, K * bits // 32), dtype=torch.int32, device="cuda")
        items.append((gu.dev(w), bits, G, gu.poison(out), torch.empty(G, device="cuda"), torch.empty(G, device="cuda")))
        host.append(w)
    call = qb.fake_quantize_weights_batch if fake else qb.quantize_pack_weights_batch
    call(items, small(ws, sum(it[2] for it in items)))
    for (_, bits, G, out, delta, q0), w in zip(items, host):
        _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, G, omp=True)
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
        if fake:
            assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.fake_quantize_weights(w, bits, G, omp=True)[1].view(np.uint32))
        else:
            assert np.array_equal(gu.words_np(out), oracle.pack(codes, bits))
    assert qb.read_status(ws) == qb.QB_OK


def test_without_a_workspace_beyond_the_ring():
    N, K, bits = 52097, 128, 3  # one unit more than the ring takes
    w = synth.weights(N, K, seed=7)
    packed = gu.poison(torch.empty((N, K * bits // 32), dtype=torch.int32, device="cuda"))
    delta, q0, status = torch.empty(1, device="cuda"), torch.empty(1, device="cuda"), torch.full((1,), 7, dtype=torch.int32, device="cuda")
    qb.quantize_pack_weights_noalloc(gu.dev(w), bits, 1, packed, delta, q0, status_out=status)
    _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, 1, omp=True)
    assert np.array_equal(gu.words_np(packed), oracle.pack(codes, bits))
    assert delta.item() == o_delta[0] and q0.item() == o_q0[0] and status.item() == qb.QB_OK


def test_nonfinite_is_reported():
    for bad in (np.nan, np.inf, -np.inf):
        for call in (qb.quantize_pack_weights, qb.fake_quantize_weights):
            ws = qb.workspace(groups=64)
            w = synth.weights(768, 768, seed=5)
            w[767, 767] = bad
            call(gu.dev(w), 4, 1, small(ws, 1))
            assert qb.read_status(ws) == qb.QB_ERR_NONFINITE
