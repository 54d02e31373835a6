"""The j-tile of compensated calls of 1.4e7 to 1.9e7 pairs: the smallest one
that leaves each of the eight CTAs per SM at most one unit (a second unit for
some of them took as long as one for all). The sums against the same pair terms
in another shape, which differ in the order of the (hi, lo) sums alone."""

import pytest

from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_i,n_j", [(7982, 2140), (10074, 1660), (8947, 1658), (2140, 7982), (3742, 3742), (4351, 4351),
                                     (10499, 1340)])
def test_one_unit_per_cta(n_i, n_j):
    cn = lib()
    torch = torch_cuda()
    ctas = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    shape = cn.cn_tune_get("dd", n_i, n_j)
    units = lambda t: -(-n_i // 64) * -(-n_j // t)  # noqa: E731
    assert shape["threads"] == 64 and units(shape["j_tile"]) <= ctas
    assert shape["j_tile"] == 32 or units(shape["j_tile"] - 32) > ctas
    di, dj = dev_tensor(synth.hernquist(n_i, 1)), dev_tensor(synth.hernquist(n_j, 2))
    a, _ = cn.cn_force_dd(di, dj, 1e-4)
    cn.cn_tune_set("dd", n_i, n_j, {"i_per_thread": 1, "threads": 128, "j_tile": 256, "stages": 4})
    try:
        b, _ = cn.cn_force_dd(di, dj, 1e-4)
    finally:
        cn.cn_tune_set("dd", n_i, n_j, None)
    assert float((a - b).norm()) <= 1e-10 * float(b.norm())
    assert cn.cn_get_device_status() == 0
