"""Token tiles of 256 or 192 for CTA pairs: the choice follows the width and the output type, since both change what a
tile costs (host arithmetic, the plan for 148 SMs without a device)."""
import pytest
import torch

import paper_1909_05840_b200 as qb
from paper_1909_05840_b200 import build as qb_build

F32, BF16, I8 = torch.float32, torch.bfloat16, torch.int8


@pytest.fixture(scope="module", autouse=True)
def built():
    qb_build.build()


def tokens(shapes, bits, out=F32, launch=0):
    arr = (qb.LinearDescC * len(shapes))()
    for d, (M, N, K) in zip(arr, shapes):
        d.M, d.N, d.K, d.bits = M, N, K, bits
    return qb.layer_linears_tile_tokens(arr, out, launch)


@pytest.mark.parametrize("bits", (2, 3, 4, 8))
@pytest.mark.parametrize("out", (F32, BF16, I8))
def test_where_both_agree(bits, out):
    # measured on either width: 1.3 rounds of 256-token tiles (192: 4 to 12 % faster), and 5.2 rounds of long tiles
    # (192: 2 to 11 % slower)
    assert tokens([(6144, 1024, 4096)], bits, out) == 192
    assert tokens([(24576, 1024, 4096)], bits, out) == 256
    assert tokens([(128, 1024, 1024)], bits, out) == 128 and tokens([(1024, 768, 768)], bits, out) == 128
    assert tokens([(300, 2304, 768), (300, 768, 768), (300, 3072, 768), (300, 768, 3072)] * 3, bits, out) == 192


def test_width_and_output_decide():
    # 192 against 256 tokens, measured: 34.7 / 35.4 us at 4 bits and 41.9 / 41.3 at 3; bfloat16 at 8 bits 31.4 / 30.5
    assert tokens([(6144, 4096, 1024)], 4) == 192 and tokens([(6144, 4096, 1024)], 3) == 256
    assert tokens([(5003, 4096, 1024)], 3) == tokens([(5003, 4096, 1024)], 8, BF16) == 256


def test_stacks_without_such_a_launch():
    assert tokens([(6144, 1024, 4096)], 4, launch=1) == 0
    assert qb.lib().qb_layer_linears_tile_tokens(None, 1, 0, 0) == 0
    assert qb.lib().qb_layer_linears_tile_tokens((qb.LinearDescC * 1)(), 1, 3, 0) == 0
