"""Digit sums of the tensor-core correlation, restated: FP32 accumulators hold
them exactly below 2^22, with the digits that the 1-D rows really have (not with
six digits of the largest magnitude each, which would not do at side 64)."""
import numpy as np
import pytest

import oracle


def digits(rows):
    """Balanced base-2^8 digits of round(rows 2^48): [6][row][column]."""
    f = np.rint(rows * 2.0 ** 48).astype(np.int64)
    out = []
    for s in range(6):
        d = ((f + 128) & 255) - 128 if s < 5 else f
        out.append(d)
        f = (f - d) >> 8
    return np.array(out)


@pytest.mark.parametrize("b,haar,pixel", [(64, False, 256), (64, True, 128), (128, False, 256)])
def test_sums_stay_below_2_22(b, haar, pixel):
    d = np.abs(digits(oracle.haar_1d(b) if haar else oracle.dct_1d(b)))
    k = b if haar else b // 2                                  # the mirror fold halves stage 2's contraction
    assert pixel * d.sum(2).max() < 2 ** 22                    # stage 1
    assert 128 * d[:, :, :k].sum((0, 2)).max() < 2 ** 22       # stage 2, six digits on a diagonal
    assert d[:5].max() <= 128 and d[5].max() <= (181 if haar else 45 if b == 64 else 32)
