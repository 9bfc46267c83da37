"""The activation quantizer's launch shapes against the oracle: one launch with the tensor in registers (a segment of
up to 1,024 elements per warp: one cluster, then several) and two passes beyond; rows of one and of several segments, rows
whose last segment is shorter, and calls that follow one another on the same workspace."""
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
    return qb.workspace(groups=64)


# 148 SMs x 16 warps = 2,368 segments in one launch, 4,736 in one wave of the second pass
@pytest.mark.parametrize("M,K", [(1, 128), (1, 65536), (7, 1024), (9, 1152), (33, 4224), (4736, 128), (4737, 128),
                                 (2368, 1152), (2369, 1152), (73, 65536), (75, 65536)])
def test_quantize_act_shapes(ws, M, K):
    for seed in (1, 2):  # the second call finds what the first left in the workspace
        x = synth.activations(M, K, seed=M + K + seed)
        if seed == 2:
            x *= np.float32(0.01)  # a smaller maximum: a slot that was not cleared would show
        xq, sc, rs = gu.gpu_quantize_act(x, ws)
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s
        assert np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
    assert qb.read_status(ws) == qb.QB_OK


# one cluster: 1 to 8 CTAs of 8 to 32 warps, the largest with 256 segments; 257 segments are beyond it
@pytest.mark.parametrize("M,K", [(8, 256), (9, 256), (17, 1024), (12, 2304), (5, 8192), (63, 768), (65, 768), (127, 640),
                                 (51, 5120), (256, 1024)])
def test_one_cluster(ws, M, K):
    for seed in (1, 2):
        x = synth.activations(M, K, seed=M + K + seed)
        x[M - 1 if seed == 1 else 0, K - 1] = 300.0  # the maximum in the last CTA or in the first
        xq, sc, rs = gu.gpu_quantize_act(x, ws)
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s
        assert np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
    x[M // 2, 1] = np.nan
    gu.gpu_quantize_act(x, ws2 := qb.workspace(groups=64))
    assert qb.read_status(ws2) == qb.QB_ERR_NONFINITE and qb.read_status(ws) == qb.QB_OK


# several clusters of 8 CTAs: 8 warps each up to 24 x 64 segments, then 16 warps, up to 2,368; 5 and 24 clusters after
# one another, so that slots of earlier calls would show
@pytest.mark.parametrize("M,K", [(257, 1024), (320, 1024), (321, 768), (150, 2304), (1536, 128), (1537, 128), (37, 65536),
                                 (592, 4096), (2368, 256), (2369, 256), (257, 128)])
def test_several_clusters(ws, M, K):
    for seed in (1, 2, 3):
        x = synth.activations(M, K, seed=M + K + seed)
        if seed != 2:
            x *= np.float32(0.01)
        x[M - 1 if seed == 1 else 0, K - 1] = 3.0 * seed  # the maximum in the last cluster or in the first
        xq, sc, rs = gu.gpu_quantize_act(x, ws)
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s
        assert np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
    x[M // 2, 1] = np.nan
    gu.gpu_quantize_act(x, ws2 := qb.workspace(groups=64))
    assert qb.read_status(ws2) == qb.QB_ERR_NONFINITE and qb.read_status(ws) == qb.QB_OK


def test_fused_call_between_batches(ws):
    # batches (two passes) and single calls (one launch) share the words that count blocks
    for rep in range(3):
        xs = [synth.activations(m, k, seed=10 * rep + m) for m, k in ((5, 256), (300, 2304), (64, 768))]
        outs = [(gu.dev(x), torch.empty(x.shape, dtype=torch.int8, device="cuda"), torch.empty(1, device="cuda"),
                 torch.empty(x.shape[0], dtype=torch.int32, device="cuda")) for x in xs]
        qb.quantize_act_batch(outs, ws)
        single = gu.gpu_quantize_act(xs[1], ws)
        for x, (_, xq, sc, rs) in zip(xs, outs):
            _, o_xq, o_s, o_rs = oracle.quantize_act(x)
            assert sc.item() == o_s and np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
        assert torch.equal(single[0], outs[1][1]) and torch.equal(single[2], outs[1][3])
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("M,K", [(64, 768), (6000, 768)])
def test_quantize_act_nonfinite_each_shape(M, K):
    for bad in (np.nan, np.inf, -np.inf):
        ws = qb.workspace(groups=64)
        x = synth.activations(M, K, seed=3)
        x[M // 2, K - 1] = bad
        gu.gpu_quantize_act(x, ws)
        assert qb.read_status(ws) == qb.QB_ERR_NONFINITE
