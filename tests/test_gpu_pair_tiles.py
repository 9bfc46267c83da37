"""CTA pairs with 192-token tiles: chosen when 256-token tiles would leave the pairs of SMs idle in the last round.
Ragged tokens and neurons, one K block to nine, every width and output type."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import synth

pytestmark = pytest.mark.gpu


# 1.1 to 1.3 rounds of 256-token tiles over 74 pairs
@pytest.mark.parametrize("bits", (2, 3, 4, 8))
@pytest.mark.parametrize("M,N,K", [(6100, 1000, 256), (6144, 1040, 1152), (5000, 1024, 128)])
def test_pairs_with_192_token_tiles(bits, M, N, K):
    ws = qb.workspace(groups=64)
    x, w, b = synth.activations(M, K, seed=M + bits), synth.weights(N, K, seed=N), synth.bias(N, seed=K)
    r = gu.check_linear(x, w, b, bits, 8, ws, rows=gu.sample_rows(M, tile=192, per_tile=2, seed=K), use_omp=True)
    args = (r["xq"], r["act_scale"], r["rowsum"], r["packed"], r["delta"], r["q0"], gu.dev(b), N, bits, 8)
    y = r["y"]
    # the narrow outputs are roundings of the fp32 value
    assert torch.equal(qb.gemm_bf16(*args, ws), y.bfloat16())
    step = (y.abs().max() / 100.0).reshape(1)
    yq = qb.gemm_i8(*args, step, ws)
    assert torch.equal(yq, torch.round(y * (torch.ones_like(step) / step)).clamp(-127, 127).to(torch.int8))
    assert qb.read_status(ws) == qb.QB_OK
