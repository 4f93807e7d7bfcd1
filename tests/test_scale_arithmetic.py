"""Kernel 1 derives ordinary scales by an approximation and one exact correction, and ordinary codes by an addition.  Both are
claimed to be bit for bit what IEEE division and conversion to integer give: compared here for every FP32 threshold of the
range in which they are used, with values at, beside and far outside every rounding boundary of the code.
"""
import numpy as np
import pytest
import torch

import paper_2605_27003_b200 as w4
from paper_2605_27003_b200 import build as pkg_build

pytestmark = pytest.mark.gpu


def pattern(x):
    return int(np.float32(x).view(np.uint32))


def test_short_scale_and_code_arithmetic_is_exact_for_every_threshold():
    pkg_build.build()
    w4.load_library()
    ctx = w4.Context(0, 128, 512, 0)
    differ = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    first, last = pattern(1e-30), pattern(1e30)
    w4.w4a4_debug_scale_arithmetic(ctx.ptr, first, last - first + 1, differ)
    assert differ.item() == 0
    for bad in ((0x7f800000, 1), (0x80000000, 1), (0x7f7fffff, 2)):
        with pytest.raises(w4.W4A4Error):
            w4.w4a4_debug_scale_arithmetic(ctx.ptr, *bad, differ)
    ctx.close()
