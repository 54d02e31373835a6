"""The compensated form's small launch shapes: parity with the FP64 oracle and
bitwise repeatability at the edges of their i-tiles, fitted j-tiles and size
range, square and not, and with zero softening."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-7  # the compensated form's


@pytest.mark.parametrize("n_i,n_j", [(1, 1), (1, 10499), (63, 33), (64, 32), (65, 31), (257, 4001), (2049, 2047),
                                     (4242, 4243), (4243, 4244), (10499, 1201), (10499, 1801), (10500, 1801)])
@pytest.mark.parametrize("eps2", [0.0, 1e-4])
def test_small_shapes(n_i, n_j, eps2):
    cn = lib()
    torch = torch_cuda()
    pi, pj = synth.hernquist(n_i, 5 + n_i), synth.hernquist(n_j, 6 + n_j)
    eps2 = float(np.float32(eps2))
    di, dj = dev_tensor(pi), dev_tensor(pj)
    a, pot = cn.cn_force_dd(di, dj, eps2, potential=True)
    b, _ = cn.cn_force_dd(di, dj, eps2)
    c, _ = cn.cn_force_dd(di, dj, eps2)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(b, c)
    # the same pair terms in another shape: only the order of the (hi, lo) sums
    # differs, each resolved to 2^-48 of its terms
    tune = {"i_per_thread": 1, "threads": 128, "j_tile": 256, "stages": 4}
    cn.cn_tune_set("dd", n_i, n_j, tune)
    try:
        d, _ = cn.cn_force_dd(di, dj, eps2)
    finally:
        cn.cn_tune_set("dd", n_i, n_j, None)
    assert float((b - d).norm()) <= 1e-10 * float(d.norm())
    rows = synth.sample_rows(n_i, min(n_i, 256), 3)
    ref, rpot = oracle.force(pi, pj, eps2, rows=rows)
    if eps2 > 0.0:  # unsoftened close pairs carry the pair term's own rounding, whatever the shape
        for x in (a, b):
            assert e_max(x.cpu().numpy()[rows], ref) <= TOL
    assert rel_pot_err(pot.cpu().numpy()[rows], rpot) <= TOL
