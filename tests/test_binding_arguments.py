"""What the Python entry refuses before it reaches the library."""
import ctypes

import pytest
import torch

import paper_1909_05840_b200 as qb

KINDS = (qb.ActDescC, qb.WeightDescC, qb.LinearDescC)


# The library reads a descriptor array as bytes: elements of another kind would become device pointers.
@pytest.mark.parametrize("call,kind", [(qb.quantize_act_batch, qb.ActDescC), (qb.quantize_pack_weights_batch, qb.WeightDescC),
                                       (qb.fake_quantize_weights_batch, qb.WeightDescC), (qb.layer_linears, qb.LinearDescC),
                                       (qb.layer_linears_bf16, qb.LinearDescC)], ids=lambda v: v.__name__)
def test_descriptor_arrays_are_typed(call, kind):
    ws = torch.zeros(4096, dtype=torch.uint8)
    for other in [k for k in KINDS if k is not kind] + [ctypes.c_uint8, ctypes.c_void_p]:
        for n in (0, 1, 7):
            with pytest.raises(ctypes.ArgumentError):
                call((other * n)(), ws)
    assert qb._descs((kind * 3)(), kind, None)._length_ == 3
    derived = type("Derived", (kind,), {})
    assert qb._descs((derived * 2)(), kind, None)._length_ == 2


@pytest.mark.gpu
def test_truth_value_that_raises():
    ws = qb.workspace(groups=256)
    packed, delta, q0 = qb.quantize_embedding(torch.rand((8, 128), device="cuda"), 4, 8, ws)
    ids = torch.zeros(3, dtype=torch.int32, device="cuda")

    class NoTruth:
        def __bool__(self):
            raise ValueError("no truth value")

    out = torch.zeros((3, 128), device="cuda")
    with pytest.raises(ValueError, match="no truth value"):
        qb.embedding_lookup(ids, packed, delta, q0, 128, 4, 8, ws, out=out, accumulate=NoTruth())
    assert not out.any()
