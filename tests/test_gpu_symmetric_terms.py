"""The three pair terms of the symmetric kernel (equal masses factored out,
general masses, and the order of operations for any range) and the mixtures
of them within a launch, at sizes around the edges of blocks, stages and
tiles, against the FP64 oracle at the plain FP32 bound."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5
SHAPES = [None, {"i_per_thread": 8, "threads": 128, "j_tile": 128, "stages": 2},
          {"i_per_thread": 4, "threads": 64, "j_tile": 32, "stages": 3}]


def _particles(kind, n):
    p = synth.plummer(n, 900 + n)
    if kind == "unequal":
        p[:, 3] *= np.random.default_rng(n).lognormal(size=n).astype(np.float32)
    elif kind == "mixed":  # equal in most stages, one other mass in the middle, a massless tail
        p[n // 2, 3] *= 5.0
        p[n - n // 5:, 3] = 0.0
    elif kind == "far":  # m r^3 and r^3 below the FP32 range, the acceleration well inside it
        p[:, :3] *= np.float32(1e14)
        p[:, 3] *= np.float32(1e28)
    elif kind == "one far":
        p[:, 3] *= np.float32(1e8)
        p[n // 3, :3] = np.float32(3e11)
    return p


@pytest.mark.parametrize("tune", SHAPES)
@pytest.mark.parametrize("kind", ["equal", "unequal", "mixed", "far", "one far"])
@pytest.mark.parametrize("n", [31, 32, 65, 1023, 1025, 4096, 6001])
def test_pair_terms(n, kind, tune):
    cn = lib()
    torch = torch_cuda()
    p = _particles(kind, n)
    eps2 = 1e24 if kind == "far" else 1e-3
    eps2 = float(np.float32(eps2))
    cn.cn_tune_set("symmetric", n, n, tune)
    try:
        a, _ = cn.cn_force_symmetric(dev_tensor(p), eps2)
        a2, pot = cn.cn_force_symmetric(dev_tensor(p), eps2, potential=True)
        torch.cuda.synchronize()
    finally:
        cn.cn_tune_set("symmetric", n, n, None)
    assert cn.cn_get_device_status() == 0
    ref, rpot = oracle.force(p, p, eps2)
    assert e_max(a.cpu().numpy(), ref) <= TOL
    assert e_max(a2.cpu().numpy(), ref) <= TOL
    assert rel_pot_err(pot.cpu().numpy(), rpot) <= TOL


def test_slots_that_grow_under_a_captured_graph():
    """A graph captured on a stream still replays after a larger call on that
    stream made the slot buffer grow."""
    cn = lib()
    torch = torch_cuda()
    p = dev_tensor(synth.plummer(5000, 1))
    big = dev_tensor(synth.plummer(40000, 2))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ref, _ = cn.cn_force_symmetric(p, 1e-3)
        torch.cuda.synchronize()
        out = torch.empty_like(ref)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            cn.cn_force_symmetric(p, 1e-3, acc_out=out)
        cn.cn_force_symmetric(big, 1e-3)
        out.zero_()
        g.replay()
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(out, ref)
