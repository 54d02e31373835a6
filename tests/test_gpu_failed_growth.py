"""A workspace that could not grow is gone, and with it every plan that held its
address: the next call of sizes that were planned before makes a new one."""

import ctypes

import pytest

from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


def _own_stream(torch):
    """A stream of its own, which no other test has used: PyTorch's come from a small pool."""
    handle = ctypes.c_uint64(0)
    assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(handle))) == 0
    return torch.cuda.ExternalStream(handle.value)


def test_call_after_a_growth_that_failed(monkeypatch):
    cn = lib()
    torch = torch_cuda()
    d = dev_tensor(synth.plummer(5000, 1))
    e = d.clone()
    big = dev_tensor(synth.hernquist(20000, 2))
    s = _own_stream(torch)
    with torch.cuda.stream(s):
        before, _ = cn.cn_force(d[:3000], e, 1e-3)
        again, _ = cn.cn_force(d[:3000], e, 1e-3)  # the plan is cached
        monkeypatch.setenv("CN_FAULT_INJECT", "alloc")
        with pytest.raises(cn.CunbodyError) as err:
            cn.cn_force(big, big[:19000].contiguous(), 1e-3)
        monkeypatch.delenv("CN_FAULT_INJECT")
        after, _ = cn.cn_force(d[:3000], e, 1e-3)
        later, _ = cn.cn_force(big, big[:19000].contiguous(), 1e-3)
    torch.cuda.synchronize()
    assert err.value.code == "CN_ERR_CUDA"
    assert torch.equal(before, again) and torch.equal(before, after)
    assert bool(torch.isfinite(later).all())
    assert cn.cn_get_device_status() == 0
