"""The row kernel (an i set against another j set; per-particle softening):
parity with the FP64 oracle at the edges of its tiles, stages and parts, with
equal, unequal and partly equal masses, positions far out and softenings of 0
among the per-particle ones; bitwise repeatable; and the calls that keep the
pair kernel."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _j_set(kind, n):
    p = synth.plummer(n, 700 + n)
    if kind == "unequal":
        p[:, 3] *= np.random.default_rng(n).lognormal(size=n).astype(np.float32)
    elif kind == "mixed":
        p[n // 3, 3] *= 7.0
        p[n - n // 6:, 3] = 0.0
    elif kind == "far":
        p[:, :3] *= np.float32(1e14)
        p[:, 3] *= np.float32(1e28)
    return p


@pytest.mark.parametrize("kind", ["equal", "unequal", "mixed", "far"])
@pytest.mark.parametrize("shape", [(128, 190003), (129, 200033), (4095, 5900), (4999, 5003), (8192, 8191), (2050, 262144)])
def test_plain_and_potential(shape, kind):
    n_i, n_j = shape
    cn = lib()
    torch = torch_cuda()
    pj = _j_set(kind, n_j)
    pi = synth.plummer(n_i, 3 + n_i)
    if kind == "far":
        pi[:, :3] *= np.float32(1e14)
    eps2 = float(np.float32(1e24 if kind == "far" else 1e-3))
    di, dj = dev_tensor(pi), dev_tensor(pj)
    a, _ = cn.cn_force(di, dj, eps2)
    again, _ = cn.cn_force(di, dj, eps2)
    a2, pot = cn.cn_force(di, dj, eps2, potential=True)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(a, again)
    rows = synth.sample_rows(n_i, 256, 9)
    ref, rpot = oracle.force(pi, pj, eps2, rows=rows)
    assert e_max(a.cpu().numpy()[rows], ref) <= TOL
    assert e_max(a2.cpu().numpy()[rows], ref) <= TOL
    assert rel_pot_err(pot.cpu().numpy()[rows], rpot) <= TOL


@pytest.mark.parametrize("zeros", [0, 1, 9])
@pytest.mark.parametrize("shape", [(4999, 5003), (129, 200033), (16385, 30600)])
def test_per_particle_softening(shape, zeros):
    cn = lib()
    torch = torch_cuda()
    n_i, n_j = shape
    pj = synth.hernquist(n_j, 31)
    pi = synth.plummer(n_i, 32)
    pi[:, 3] = np.random.default_rng(33).uniform(1e-4, 5e-2, n_i).astype(np.float32)
    if zeros:
        pi[::n_i // zeros, 3] = 0.0
        pi[0, :3] = pj[7, :3]  # eps2_i = 0 on top of a j particle
    a, pot = cn.cn_force_eps_i(dev_tensor(pi), dev_tensor(pj), potential=True)
    a2, _ = cn.cn_force_eps_i(dev_tensor(pi), dev_tensor(pj))
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    rows = np.unique(np.concatenate([synth.sample_rows(n_i, 256, 34), np.flatnonzero(pi[:, 3] == 0.0)]))
    ref, rpot = oracle.force_eps_i(pi, pj, rows=rows)
    for x in (a, a2):
        assert np.all(np.isfinite(x.cpu().numpy()))
        assert e_max(x.cpu().numpy()[rows], ref) <= TOL
    assert rel_pot_err(pot.cpu().numpy()[rows], rpot) <= TOL


def test_workspaces_and_tunes():
    cn = lib()
    torch = torch_cuda()
    di, dj = dev_tensor(synth.plummer(3000, 1)), dev_tensor(synth.plummer(20000, 2))
    rows, _ = cn.cn_force(di, dj, 1e-3)
    ws = torch.empty(cn.cn_workspace_bytes("f32", 3000, 20000), dtype=torch.uint8, device="cuda")
    same, _ = cn.cn_force_ws(di, dj, 1e-3, ws)
    cn.cn_tune_set("f32", 3000, 20000, cn.cn_tune_get("f32", 3000, 20000))
    try:
        pair, _ = cn.cn_force(di, dj, 1e-3)
    finally:
        cn.cn_tune_set("f32", 3000, 20000, None)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    assert torch.equal(rows, same) and not torch.equal(rows, pair)
    assert e_max(rows.cpu().numpy(), pair.cpu().numpy().astype(np.float64)) <= 2 * TOL
