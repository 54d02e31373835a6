"""The sums that a CTA hands over at the end of its part of a row keep both
words: a term of 2^-26 of the sum beside it survives until another CTA's part
cancels the sum."""

import numpy as np
import pytest

from gpu_common import dev_tensor, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk_units", [0, 3])  # one band of rows, bands of three
def test_small_term_beside_a_sum_that_cancels(chunk_units):
    cn = lib()
    n = 20000
    # 152 CTAs at about 82 blocks of 32 records: blocks 30 and 60 of row 0 are the first one's, 600 is not
    p = np.zeros((n, 4), dtype=np.float32)
    for block, x, m in ((30, 1.0, 1.0), (60, 1.0, 2.0 ** -26), (600, -1.0, 1.0)):
        p[32 * block, 0] = x
        p[32 * block, 3] = m
    cn.cn_tune_set("symmetric", n, n, {"i_per_thread": 2, "threads": 256, "j_tile": 128, "stages": 3, "ctas_per_sm": 1,
                                       "chunk_units": chunk_units})
    try:
        a, _ = cn.cn_force_symmetric(dev_tensor(p), 1.0)
    finally:
        cn.cn_tune_set("symmetric", n, n, None)
    assert cn.cn_get_device_status() == 0
    a = a.cpu().numpy().astype(np.float64)[p[:, 0] == 0.0]
    # r^-3 of the pair term is the same number for all three: only its own error remains (under 2^-20)
    want = 2.0 ** -1.5 * 2.0 ** -26
    assert np.all(a[:, 1:] == 0.0) and np.all(np.abs(a[:, 0] - want) <= 2.0 ** -20 * want)
