"""A workspace asked for one size serves every smaller call of the compensated
form, whatever j-tile is fitted to it."""

import numpy as np
import pytest

from gpu_common import dev_tensor, e_max, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("potential", [False, True])
@pytest.mark.parametrize("size,parts", [((1000, 1000), [(900, 900), (64, 1000), (999, 33)]),
                                        ((3300, 3300), [(1500, 1500), (2000, 2000), (2600, 2600), (3000, 1800)]),
                                        ((100, 11000), [(100, 10400), (65, 7000)]),
                                        ((6144, 6144), [(4400, 4400), (5000, 5000), (6000, 6000)]),
                                        ((20000, 30), [(10400, 30), (700, 29)])])
def test_parts_of_a_set(size, parts, potential):
    cn = lib()
    torch = torch_cuda()
    pi, pj = dev_tensor(synth.plummer(size[0], 1)), dev_tensor(synth.hernquist(size[1], 2))
    ws = torch.empty(cn.cn_workspace_bytes("dd_pot" if potential else "dd", *size), dtype=torch.uint8, device="cuda")
    for n_i, n_j in [size] + parts:
        a, _ = cn.cn_force_dd_ws(pi[:n_i], pj[:n_j], 1e-3, ws, potential=potential)
        b, _ = cn.cn_force_dd(pi[:n_i], pj[:n_j], 1e-3, potential=potential)
        torch.cuda.synchronize()
        assert torch.equal(a, b)
    assert cn.cn_get_device_status() == 0
