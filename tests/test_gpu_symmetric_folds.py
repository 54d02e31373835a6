"""Sums of the symmetric force and jerk forms of mid-size sets add at most 128
records in FP32 registers before they go into (hi, lo) sums: there the pair
kernel's chains are short too.

A heavy record opens the first CTA's part, 255 light ones follow, each below
half an ulp of the heavy one's term: behind it in one chain of additions they
are lost, in the next one they count. The heavy one alone gives the value that
the light ones add to, with the same error of the pair term."""

import numpy as np
import pytest

from gpu_common import dev_tensor, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,n", [("force", 12000), ("force", 18000), ("pot", 12000), ("pot", 20000),
                                    ("symmetric", 25001), ("jerk", 9000), ("jerk", 15000)])
def test_light_records_behind_a_heavy_one(form, n):
    cn = lib()
    # two masses in turn: those of a stage that were all equal would be summed apart
    light = np.where(np.arange(255) % 2, 0.7, 0.6).astype(np.float32) * np.float32(2.0 ** -25)

    def run(mass):
        p = np.zeros((n, 4), dtype=np.float32)
        p[:256, :3] = 1.0
        p[0, 3] = 1.0
        p[1:256, 3] = mass
        d = dev_tensor(p)
        if form == "jerk":
            v = dev_tensor(np.zeros((n, 4), dtype=np.float32))
            out = cn.cn_force_jerk(d, v, d, v, 1.0)[0]
        elif form == "symmetric":
            out = cn.cn_force_symmetric(d, 1.0)[0]
        else:
            a, phi = cn.cn_force(d, d, 1.0, potential=form == "pot")
            out = a if phi is None else phi
        return out.cpu().numpy()[256:400].astype(np.float64)  # at the origin, in the first tile

    more = run(light) / run(0.0) - 1.0
    assert cn.cn_get_device_status() == 0
    # at most the 127 behind the heavy record in its chain are lost; the results' own roundings: 2^-23
    assert np.all(np.abs(more - light.sum(dtype=np.float64)) <= light[:127].sum(dtype=np.float64) + 2.0 ** -23)
