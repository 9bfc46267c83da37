"""A call of two launches of which the second never ran (refused, say) leaves a workspace that serves the next call.  Such
a call is made here as a graph that holds the first launch alone."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


def run_first_launch(call):
    """Enqueue the first kernel of ``call`` alone."""
    rt = pytest.importorskip("cuda.bindings.runtime")

    def ok(result):
        assert int(result[0]) == 0, result[0]
        return result[1] if len(result) == 2 else result[1:]

    call()  # whatever is set up once
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    graph = rt.cudaGraph_t(g.raw_cuda_graph())
    count = ok(rt.cudaGraphGetNodes(graph))[1]
    nodes = ok(rt.cudaGraphGetNodes(graph, count))[0]
    roots = {int(n) for n in ok(rt.cudaGraphGetRootNodes(graph, ok(rt.cudaGraphGetRootNodes(graph))[1]))[0]}
    assert count == 2 and len(roots) == 1, "the call has another shape than this test is made for"
    for n in nodes:
        if int(n) not in roots:
            ok((*rt.cudaGraphDestroyNode(n), None))
    run = ok(rt.cudaGraphInstantiate(graph, 0))
    ok((*rt.cudaGraphLaunch(run, torch.cuda.current_stream().cuda_stream), None))
    torch.cuda.synchronize()
    ok((*rt.cudaGraphExecDestroy(run), None))


@pytest.mark.parametrize("reps", (1, 3))
def test_activations(reps):
    ws = qb.workspace(groups=64)
    big = gu.dev(synth.activations(6000, 768, seed=1) * np.float32(100.0))
    out = (torch.empty((6000, 768), dtype=torch.int8, device="cuda"), torch.empty(1, device="cuda"),
           torch.empty(6000, dtype=torch.int32, device="cuda"))
    for _ in range(reps):
        run_first_launch(lambda: qb.quantize_act(big, ws, *out))
    for M, K in ((6000, 768), (4737, 128), (6000, 768)):
        x = synth.activations(M, K, seed=M)
        xq, sc, rs = gu.gpu_quantize_act(x, ws)
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s
        assert np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
    assert qb.read_status(ws) == qb.QB_OK


def test_activation_batches():
    ws = qb.workspace(groups=64)

    def items(xs):
        return [(gu.dev(x), torch.empty(x.shape, dtype=torch.int8, device="cuda"), torch.empty(1, device="cuda"),
                 torch.empty(x.shape[0], dtype=torch.int32, device="cuda")) for x in xs]

    xs = [synth.activations(m, k, seed=m) for m, k in ((5, 256), (300, 2304), (64, 768))]
    big = qb.make_act_desc_array(first := items([x * np.float32(50.0) for x in xs]))
    run_first_launch(lambda: qb.quantize_act_batch(big, ws))
    small = items(xs)
    qb.quantize_act_batch(small, ws)
    for x, (_, xq, sc, rs) in zip(xs, small):
        _, o_xq, o_s, o_rs = oracle.quantize_act(x)
        assert sc.item() == o_s and np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
    assert len(first) == 3 and qb.read_status(ws) == qb.QB_OK


def test_embedding_tables():
    ws = qb.workspace(groups=4096)
    rng = np.random.default_rng(3)
    e = (rng.standard_normal((700, 256)) * 0.02).astype(np.float32)
    big = gu.dev(e * np.float32(50.0))
    packed = torch.empty((700, 256 * 4 // 32), dtype=torch.int32, device="cuda")
    run_first_launch(lambda: qb.quantize_embedding(big, 4, 16, ws, packed=packed))
    for _ in range(2):
        packed, delta, q0 = qb.quantize_embedding(gu.dev(e), 4, 16, ws)
        _, codes, o_delta, o_q0 = oracle.quantize_embedding(e, 4, 16)
        assert np.array_equal(gu.words_np(packed), oracle.pack(codes, 4))
        assert np.array_equal(delta.cpu().numpy(), o_delta) and np.array_equal(q0.cpu().numpy(), o_q0)
    assert qb.read_status(ws) == qb.QB_OK
