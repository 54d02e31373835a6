"""The autotuner against calls that take the row or the symmetric kernel by
default: it times that default, and a shape found for calls of two sets does
not keep one set against itself out of the symmetric kernel, also after a
round trip through a tuning file."""

import pytest

from gpu_common import dev_tensor, lib
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["f32", "f32_pot"])
def test_row_kernel_stays_where_it_is_the_fastest(variant):
    cn = lib()
    n_i, n_j, pot = 1024, 65536, variant == "f32_pot"
    di, dj = dev_tensor(synth.plummer(n_i, 1)), dev_tensor(synth.plummer(n_j, 2))
    before, _ = cn.cn_force(di, dj, 1e-3, potential=pot)
    cn.cn_autotune(variant, di, dj, 1e-3, reps=5)
    try:
        after, _ = cn.cn_force(di, dj, 1e-3, potential=pot)
    finally:
        cn.cn_tune_set(variant, n_i, n_j, None)
    assert bool((after == before).all())


def test_two_sets_do_not_decide_for_one(tmp_path):
    cn = lib()
    n = 12001
    d, e = dev_tensor(synth.plummer(n, 3)), dev_tensor(synth.plummer(n, 4))
    one, _ = cn.cn_force(d, d, 1e-3)
    need = cn.cn_workspace_bytes("f32", n, n)
    cn.cn_autotune("f32", d, e, 1e-3, reps=2)
    try:
        tuned = cn.cn_tune_get("f32", n, n)
        two, _ = cn.cn_force(d, e, 1e-3)
        after, _ = cn.cn_force(d, d, 1e-3)
        assert bool((after == one).all()) and cn.cn_workspace_bytes("f32", n, n) == need
        path = str(tmp_path / "tune.json")
        cn.cn_tune_save(path)
        cn.cn_tune_set("f32", n, n, None)
        cn.cn_tune_load(path)
        assert cn.cn_tune_get("f32", n, n) == tuned
        assert bool((cn.cn_force(d, d, 1e-3)[0] == one).all()) and bool((cn.cn_force(d, e, 1e-3)[0] == two).all())
        # the same shape stored by hand is meant for every call of the class
        cn.cn_tune_set("f32", n, n, tuned)
        assert not bool((cn.cn_force(d, d, 1e-3)[0] == one).all())
    finally:
        cn.cn_tune_set("f32", n, n, None)
    assert cn.cn_get_device_status() == 0
