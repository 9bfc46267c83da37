"""The tensor-core probe measures the instruction, not its issue: half the tokens take half the time."""
import pytest

import gpu_util as gu
import paper_1909_05840_b200 as qb

pytestmark = pytest.mark.gpu


def test_rate_does_not_depend_on_the_tokens():
    gu.ensure_built()
    tops = {t: qb.probe_i8_mma(t, 20000) for t in (128, 256)}
    # 2 cycles per token and K block at either width, so half at 128; an issue-bound probe takes as long for
    # both widths, so the line lies half-way between (a ratio of 0.7 instead of 1 or 0.5)
    assert tops[128][1] < 0.7 * tops[256][1], tops
    assert tops[128][0] > 0.7 * tops[256][0], tops
