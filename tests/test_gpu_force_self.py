"""cn_force on one set against itself takes the symmetric kernel above 4096
particles: parity with the FP64 oracle on both sides of that line, and the
calls that keep the one-sided kernel (another copy of the set, a registered
tune, zero softening, a workspace that holds no slots, a capture or a memory
limit that does not let the slots grow)."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.mark.parametrize("potential", [False, True])
@pytest.mark.parametrize("n", [4096, 4097, 5999, 6000, 12001, 24577])
def test_parity_across_the_line(n, potential):
    cn = lib()
    torch = torch_cuda()
    p = synth.hernquist(n, n) if n % 2 else synth.plummer(n, n)
    d = dev_tensor(p)
    a, pot = cn.cn_force(d, d, 1e-3, potential=potential)
    b, _ = cn.cn_force(d, d.clone(), 1e-3, potential=potential)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    rows = synth.sample_rows(n, 1024, 3)
    ref, rpot = oracle.force(p, p, 1e-3, rows=rows)
    assert e_max(a.cpu().numpy()[rows], ref) <= TOL
    assert e_max(b.cpu().numpy()[rows], ref) <= TOL
    if potential:
        assert rel_pot_err(pot.cpu().numpy()[rows], rpot) <= TOL


def test_calls_that_keep_the_one_sided_kernel(monkeypatch):
    cn = lib()
    torch = torch_cuda()
    n = 9000
    p = synth.plummer(n, 2)
    d = dev_tensor(p)
    one, _ = cn.cn_force(d, d.clone(), 1e-3)
    both, _ = cn.cn_force(d, d, 1e-3)
    shape = cn.cn_tune_get("f32", n, n)
    cn.cn_tune_set("f32", n, n, shape)
    try:
        tuned, _ = cn.cn_force(d, d, 1e-3)
    finally:
        cn.cn_tune_set("f32", n, n, None)
    assert torch.equal(tuned, one) and not torch.equal(both, one)
    # a caller's workspace: the bytes asked for, and those of the one-sided kernel alone
    need = cn.cn_workspace_bytes("f32", n, n)
    full, _ = cn.cn_force_ws(d, d, 1e-3, torch.empty(need, dtype=torch.uint8, device="cuda"))
    small = cn.cn_workspace_bytes("f32", n, n - 1)
    assert small < need
    less, _ = cn.cn_force_ws(d, d, 1e-3, torch.empty(small + (1 << 16), dtype=torch.uint8, device="cuda"))
    assert torch.equal(full, both) and torch.equal(less, one)
    # a fresh stream: with no memory for the slots nothing is left behind, and later calls have them
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        cn.cn_force(d, d.clone(), 1e-3)
        monkeypatch.setenv("CN_FAULT_INJECT", "alloc")
        limited, _ = cn.cn_force(d, d, 1e-3)
        monkeypatch.setenv("CN_FAULT_INJECT", "capture")
        captured, _ = cn.cn_force(d, d, 1e-3)
        monkeypatch.delenv("CN_FAULT_INJECT")
        later, _ = cn.cn_force(d, d, 1e-3)
    torch.cuda.synchronize()
    assert torch.equal(limited, one) and torch.equal(captured, one) and torch.equal(later, both)
    zero, _ = cn.cn_force(d, d, 0.0)
    ref, _ = oracle.force(p, p, 0.0, rows=np.arange(300), potential=False)
    torch.cuda.synchronize()
    assert e_max(zero.cpu().numpy()[:300], ref) <= TOL
    assert cn.cn_get_device_status() == 0


def test_first_call_inside_a_capture():
    cn = lib()
    torch = torch_cuda()
    n = 7000
    d = dev_tensor(synth.plummer(n, 4))
    cn.cn_tune_set("f32", n, n, cn.cn_tune_get("f32", n, n))
    one, _ = cn.cn_force(d, d, 1e-3)  # the one-sided kernel
    cn.cn_tune_set("f32", n, n, None)
    s = torch.cuda.Stream()
    out = torch.zeros((n, 3), device="cuda")
    with torch.cuda.stream(s):
        cn.cn_force(d, d.clone(), 1e-3)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            cn.cn_force(d, d, 1e-3, acc_out=out)
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, one)
