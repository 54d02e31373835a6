"""Ensembles whose plan takes the symmetric form: clusters around the edges of
blocks and tiles (single particles and empty ones among them), equal and
unequal masses, with and without the potential, against the FP64 oracle; and
a caller's workspace without room for the slots, which takes the one-sided
kernel."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5
SIZES = {"large": [9000, 8191, 2049, 0, 4096, 1, 513, 12000, 31], "mid": [3000, 2500, 1025, 1024, 1023, 2, 0, 3100] * 12}


def _ensemble(kind, unequal):
    sizes = SIZES[kind]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    make = synth.hernquist if unequal else synth.plummer
    rec = np.concatenate([make(m, 40 + c) for c, m in enumerate(sizes) if m])
    eps2 = np.array([np.float32(0.01 + 1e-3 * (c % 5)) for c in range(len(sizes))], dtype=np.float32)
    return rec, offs, eps2


@pytest.mark.parametrize("potential", [False, True])
@pytest.mark.parametrize("unequal", [False, True])
@pytest.mark.parametrize("kind", ["large", "mid"])
def test_parity(kind, unequal, potential):
    cn = lib()
    torch = torch_cuda()
    rec, offs, eps2 = _ensemble(kind, unequal)
    plan = cn.BatchPlan(offs, eps2, potential=potential)
    d = dev_tensor(rec)
    acc, pot = plan.run(d)
    again, _ = plan.run(d)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(acc, again)
    a = acc.cpu().numpy()
    for c in range(len(offs) - 1):
        lo, hi = int(offs[c]), int(offs[c + 1])
        if hi - lo < 2:
            assert np.all(a[lo:hi] == 0)
            continue
        rows = synth.sample_rows(hi - lo, 256, c)
        ref, rpot = oracle.force(rec[lo:hi], rec[lo:hi], eps2[c], rows=rows)
        assert e_max(a[lo:hi][rows], ref) <= TOL, c
        if potential:
            assert rel_pot_err(pot.cpu().numpy()[lo:hi][rows], rpot) <= TOL, c
    plan.close()


def test_a_workspace_without_slots_takes_the_one_sided_kernel():
    cn = lib()
    torch = torch_cuda()
    rec, offs, eps2 = _ensemble("large", False)
    d = dev_tensor(rec)
    plan = cn.BatchPlan(offs, eps2)
    both, _ = plan.run(d)
    full, _ = plan.run(d, workspace=plan.new_workspace())
    one_plan = cn.BatchPlan(offs, eps2, tune={"i_per_thread": 4, "threads": 64, "j_tile": 256, "stages": 4})
    ref, _ = one_plan.run(d)
    few = torch.zeros(plan.workspace_bytes - 256, dtype=torch.uint8, device="cuda")
    less, _ = plan.run(d, workspace=few)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(full, both) and not torch.equal(less, both)
    assert e_max(less.cpu().numpy(), ref.cpu().numpy().astype(np.float64)) <= 2 * TOL
    with pytest.raises(cn.CunbodyError):
        plan.run(d, workspace=few[:256])
    plan.close()
    one_plan.close()
