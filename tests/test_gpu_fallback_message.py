"""A call that succeeds without a step it can do without (slots of the symmetric
form, segments of the row kernel) leaves no error message behind."""

import ctypes
import threading

import numpy as np
import pytest

from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


def _own_stream(torch):
    """A stream of its own, which no other test has used: PyTorch's come from a small pool."""
    handle = ctypes.c_uint64(0)
    assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(handle))) == 0
    return torch.cuda.ExternalStream(handle.value)


@pytest.mark.parametrize("fault", ["alloc", "capture"])
@pytest.mark.parametrize("form", ["force", "rows", "jerk", "ensemble"])
def test_no_message_after_a_fallback(monkeypatch, form, fault):
    cn = lib()
    torch = torch_cuda()
    n = 6000
    d, v = dev_tensor(synth.plummer(n, 1)), dev_tensor(synth.plummer_velocities(n, 2))
    j = dev_tensor(synth.plummer(40000, 3))
    plan = cn.BatchPlan(np.array([0, n], dtype=np.int64), np.full(1, 1e-3, dtype=np.float32))
    wide = cn.BatchPlan(np.array([0, n], dtype=np.int64), np.full(1, 1e-3, dtype=np.float32),
                        tune={"i_per_thread": 8, "threads": 256, "j_tile": 128, "stages": 3})
    got = []

    def work():  # a thread of its own has no earlier message
        s = _own_stream(torch)
        with torch.cuda.stream(s):
            cn.cn_force_eps_i(j, j[:500].contiguous())  # the one-sided workspaces alone
            wide.run(d)
            if form == "rows":
                cn.cn_tune_set("f32", 1000, 40000, cn.cn_tune_get("f32", 1000, 40000))
                cn.cn_force(d[:1000], j, 1e-3)
                cn.cn_tune_set("f32", 1000, 40000, None)
            else:
                cn.cn_force(d, d.clone(), 1e-3)
            cn.cn_force_jerk(d, v, d.clone(), v, 1e-3)
            cn.cn_force_jerk(j[:9000], j[:9000], j[:9000].clone(), j[:9000], 1e-3)
            monkeypatch.setenv("CN_FAULT_INJECT", fault)
            try:
                if form == "force":
                    cn.cn_force(d, d, 1e-3)
                elif form == "rows":
                    cn.cn_force(d[:1000], j, 1e-3)
                elif form == "jerk":
                    cn.cn_force_jerk(d, v, d, v, 1e-3)
                else:
                    plan.run(d)
            except cn.CunbodyError as e:
                got.append(e)
            finally:
                monkeypatch.delenv("CN_FAULT_INJECT")
            got.append(cn.cn_last_error_message())

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    plan.close()
    wide.close()
    assert got == [""]
    assert cn.cn_get_device_status() == 0
