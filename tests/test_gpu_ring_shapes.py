"""The weight quantizer's single-read path for groups too large for a cluster's registers, against the oracle: groups
of one to eleven rounds of 148 chunks (of 32 units of 128 weights), last chunks of any length, several groups per
matrix, packing and fake quantization, a batch of mixed widths; and the two passes just beyond."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ws():
    return qb.workspace(groups=4096)


# units per group: 2,305 (73 chunks), 148 chunks exactly, one more, 32 k + 1, 11 * 148 chunks (the last size that
# fits) and one unit more (two passes)
@pytest.mark.parametrize("N,K,groups", [(2305, 128, 1), (768, 768, 1), (4736, 128, 1), (4737, 128, 1), (5210, 256, 2),
                                        (3072, 768, 1), (52096, 128, 1), (52097, 128, 1)])
def test_large_groups(ws, N, K, groups):
    w = synth.weights(N, K, seed=N + K)
    for bits in (2, 3, 4, 8):
        packed, delta, q0 = gu.gpu_quantize_weights(w, bits, groups, ws)
        _, codes, o_delta, o_q0 = oracle.quantize_weights(w, bits, groups, omp=True)
        assert np.array_equal(gu.words_np(packed), oracle.pack(codes, bits)), bits
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
    wq, delta, q0 = qb.fake_quantize_weights(gu.dev(w), 4, groups, ws)
    st, o_wq, o_delta, o_q0 = oracle.fake_quantize_weights(w, 4, groups)
    assert np.array_equal(wq.cpu().numpy().view(np.uint32), o_wq.view(np.uint32))
    assert qb.read_status(ws) == qb.QB_OK


def test_mixed_batch_equals_single_calls(ws):
    shapes = [(768, 768, 3, 1), (2304, 768, 2, 3), (3072, 768, 8, 1), (768, 3072, 4, 1), (1111, 640, 3, 1), (768, 768, 4, 768)] * 3
    items, keep = [], []
    for i, (N, K, bits, G) in enumerate(shapes):
        w = gu.dev(synth.weights(N, K, seed=i))
        items.append((w, bits, G, torch.empty((N, K * bits // 32), dtype=torch.int32, device="cuda"),
                      torch.empty(G, device="cuda"), torch.empty(G, device="cuda")))
    for _ in range(3):
        for it in items:
            it[3].fill_(-1)
        qb.quantize_pack_weights_batch(items, ws)
        for w, bits, G, packed, delta, q0 in items:
            p, d, z = qb.quantize_pack_weights(w, bits, G, ws)
            assert torch.equal(p, packed) and torch.equal(d, delta) and torch.equal(z, q0)
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_is_reported(bad):
    ws = qb.workspace(groups=64)
    w = synth.weights(3072, 768, seed=5)
    w[3071, 767] = bad
    gu.gpu_quantize_weights(w, 4, 1, ws)
    assert qb.read_status(ws) == qb.QB_ERR_NONFINITE


def test_workspace_without_room_for_the_slots():
    # 8 bytes per group are enough: the two passes serve the call
    G = 40
    ws = qb.workspace(groups=4096)
    small = ws[:((256 + 8 * G + 255) // 256) * 256]
    w = synth.weights(768 * G, 768, seed=6).reshape(768 * G, 768)
    packed = torch.empty((768 * G, 96), dtype=torch.int32, device="cuda")
    delta, q0 = torch.empty(G, device="cuda"), torch.empty(G, device="cuda")
    qb.quantize_pack_weights(gu.dev(w), 4, G, small, packed=packed, delta=delta, q0=q0)
    p, d, z = qb.quantize_pack_weights(gu.dev(w), 4, G, ws)
    assert torch.equal(p, packed) and torch.equal(d, delta) and torch.equal(z, q0)
