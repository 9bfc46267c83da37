"""Python threads: a call that blocks in the library (a full launch queue) leaves the interpreter to the others; threads with
a stream and a workspace each run the kernels that need all their blocks resident side by side."""
import threading
import time

import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


def test_blocking_call_leaves_the_interpreter_to_other_threads():
    ws = qb.workspace(groups=64)
    item = (gu.dev(synth.activations(8, 128, seed=1)), torch.empty((8, 128), dtype=torch.int8, device="cuda"),
            torch.empty(1, device="cuda"), torch.empty(8, dtype=torch.int32, device="cuda"))
    arr = qb.make_act_desc_array([item])
    calls = {"single": lambda: qb.quantize_act(item[0], ws, *item[1:]), "over descriptors": lambda: qb.quantize_act_batch(arr, ws)}
    for call in calls.values():
        call()
    torch.cuda.synchronize()
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.001)

    other = threading.Thread(target=tick)
    other.start()
    try:
        for name, call in calls.items():
            torch.cuda._sleep(1_000_000_000)  # half a second: the launches behind it fill the queue
            for _ in range(20000):
                t0 = time.perf_counter()
                call()
                t1 = time.perf_counter()
                if t1 - t0 > 0.1:
                    break
            assert t1 - t0 > 0.1, f"{name}: no call blocked"
            during = [t for t in ticks if t0 <= t <= t1]
            # a tick per millisecond; ten leave room for a busy machine, a held lock lets two through at most
            assert len(during) > 10, f"{name}: {len(during)} ticks in {t1 - t0:.2f} s"
            torch.cuda.synchronize()
    finally:
        stop.set()
        other.join()
    assert qb.read_status(ws) == qb.QB_OK


def test_streams_side_by_side():
    M, N, K, bits = 2368, 768, 768, 4
    xs = [synth.activations(M, K, seed=i) * np.float32(1 + i) for i in range(2)]
    weights = [synth.weights(N, K, seed=10 + i) * np.float32(1 + i) for i in range(2)]
    inputs = [(gu.dev(x), gu.dev(w), qb.workspace(groups=4096)) for x, w in zip(xs, weights)]
    torch.cuda.synchronize()
    results, errors = [[], []], []
    start = threading.Barrier(2)

    def work(i):
        try:
            x, w, ws = inputs[i]
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for rep in range(25):
                    act = qb.quantize_act(x, ws)  # several clusters, all resident
                    pack = qb.quantize_pack_weights(w, bits, 1, ws)  # the ring: every SM
                    y = qb.gemm(*act, *pack, None, N, bits, 1, ws)
                    if rep % 8 == 0:
                        results[i].append((act, pack, y))
                torch.cuda.current_stream().synchronize()
        except Exception as e:  # noqa: BLE001 (reported below, in the test's own thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        assert qb.read_status(inputs[i][2]) == qb.QB_OK
        _, o_xq, o_s, o_rs = oracle.quantize_act(xs[i])
        _, codes, o_delta, o_q0 = oracle.quantize_weights(weights[i], bits, 1)
        for (xq, sc, rs), (packed, delta, q0), y in results[i]:
            assert sc.item() == o_s and np.array_equal(xq.cpu().numpy(), o_xq) and np.array_equal(rs.cpu().numpy(), o_rs)
            assert np.array_equal(gu.words_np(packed), oracle.pack(codes, bits))
            assert delta.item() == o_delta[0] and q0.item() == o_q0[0]
            assert torch.equal(y, results[i][0][2])
        o_acc = oracle.int_gemm(o_xq[:40], codes)
        gu.assert_y_close(results[i][0][2][:40].cpu().numpy(),
                          oracle.dequant_epilogue(o_acc, o_rs[:40], o_s, o_delta, o_q0, None, bits, 1))
