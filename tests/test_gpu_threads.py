"""Python threads: a call that blocks in the library (a full launch queue) leaves the interpreter to the others."""
import threading
import time

import pytest
import torch

import gpu_util as gu
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
