"""The embedding and straight-through kernels at the sizes where their loops begin and end, against the oracle: fewer
rows than a block reads side by side, one row more or less than a round of rows in flight, groups of one and of all
columns, group boundaries inside a warp's units, in-place gradients."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ws():
    return qb.workspace(groups=4096)


# D = 128 .. 4096: 16 rows to one row side by side; rows around 2 * 148 * slots * 8
@pytest.mark.parametrize("V,D,groups", [(1, 128, 128), (3, 256, 1), (17, 128, 8), (592, 768, 48), (593, 768, 6), (4737, 768, 1),
                                        (2368, 1024, 1024), (299, 4096, 4096), (300, 2048, 64), (5, 4096, 1)])
def test_embedding_shapes(ws, V, D, groups):
    rng = np.random.default_rng(V * 7 + D)
    e = (rng.standard_normal((V, D)) * 0.02).astype(np.float32)
    for bits in (2, 3, 4, 8):
        packed, delta, q0 = qb.quantize_embedding(gu.dev(e), bits, groups, ws)
        st, codes, o_delta, o_q0 = oracle.quantize_embedding(e, bits, groups)
        assert np.array_equal(gu.words_np(packed), oracle.pack(codes, bits)), bits
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
        for T in (1, 5, 4 * 148 * 2 + 1):
            ids = rng.integers(0, V, T).astype(np.int32)
            ref = oracle.embedding_lookup(ids, codes, groups, o_delta, o_q0)
            out = qb.embedding_lookup(gu.dev(ids), packed, delta, q0, D, bits, groups, ws)
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))
            ref = oracle.embedding_lookup(ids, codes, groups, o_delta, o_q0, out=ref)
            qb.embedding_lookup(gu.dev(ids), packed, delta, q0, D, bits, groups, ws, out=out, accumulate=True)
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    assert qb.read_status(ws) == qb.QB_OK


@pytest.mark.parametrize("N,K,groups", [(1, 128, 1), (3, 128, 3), (31, 128, 31), (33, 384, 11), (257, 1152, 257), (768, 768, 1), (96, 16384, 12)])
def test_ste_shapes(N, K, groups):
    rng = np.random.default_rng(N + K)
    w = (rng.standard_normal((N, K)) * 0.1).astype(np.float32)
    g = rng.standard_normal((N, K)).astype(np.float32)
    lo = (-0.1 - 0.05 * rng.random(groups)).astype(np.float32)
    hi = (0.1 + 0.05 * rng.random(groups)).astype(np.float32)
    w[0, 0] = lo[0]  # both ends pass
    w[-1, -1] = hi[-1]
    ref = oracle.ste_backward(g, w, groups, lo, hi)
    gt = gu.dev(g)
    out = qb.ste_backward(gt, gu.dev(w), groups, gu.dev(lo), gu.dev(hi))
    assert np.array_equal(out.cpu().numpy(), ref)
    qb.ste_backward(gt, gu.dev(w), groups, gu.dev(lo), gu.dev(hi), grad_w=gt)  # in place
    assert np.array_equal(gt.cpu().numpy(), ref)
