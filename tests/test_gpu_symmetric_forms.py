"""The force-jerk and adjoint forms of one set against itself take the
symmetric kernel above 2048 particles: parity with the FP64 oracle at sizes
around the line and the edges of blocks and tiles, equal and unequal masses,
positions far out, coincident particles; and the calls that keep the
one-sided kernel. Bounds as in the tests of the two forms."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib, rel_pot_err, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL_ACC, TOL_JERK = 1e-5, 2e-5
TOL_POS, TOL_MASS = 1.5e-5, 1e-6


def _set(kind, n):
    p = synth.plummer(n, 300 + n)
    if kind == "unequal":
        p[:, 3] *= np.random.default_rng(n).lognormal(size=n).astype(np.float32)
    elif kind == "coincident":
        p[n - 40:] = p[100:140]
    elif kind == "far":
        p[:, :3] *= np.float32(1e12)
        p[:, 3] *= np.float32(1e24)
    return p


@pytest.mark.parametrize("kind", ["equal", "unequal", "coincident", "far"])
@pytest.mark.parametrize("n", [2048, 2049, 4999, 5003, 20001])
def test_jerk_of_one_set(n, kind):
    cn = lib()
    torch = torch_cuda()
    p, v = _set(kind, n), synth.plummer_velocities(n, 400 + n)
    eps2 = float(np.float32(1e20 if kind == "far" else 1e-3))
    d, dv = dev_tensor(p), dev_tensor(v)
    a, j, pot = cn.cn_force_jerk(d, dv, d, dv, eps2, potential=True)
    a2, j2, _ = cn.cn_force_jerk(d, dv, d, dv, eps2)
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    rows = synth.sample_rows(n, 1024, 5)
    ra, rj, rp = oracle.force_jerk(p[rows], v[rows], p, v, eps2)
    for x in (a, a2):
        assert e_max(x.cpu().numpy()[rows], ra) <= TOL_ACC
    for x in (j, j2):
        assert e_max(x.cpu().numpy()[rows], rj) <= TOL_JERK
    assert rel_pot_err(pot.cpu().numpy()[rows], rp) <= TOL_ACC


@pytest.mark.parametrize("kind", ["equal", "unequal", "coincident"])
@pytest.mark.parametrize("n", [2048, 2049, 6501, 9999])
def test_adjoint(n, kind):
    cn = lib()
    torch = torch_cuda()
    p, w = _set(kind, n), synth.adjoint_weights(n, 500 + n)
    gp, gm = cn.cn_force_adjoint(dev_tensor(p), 0.01, dev_tensor(w))
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    rows = synth.sample_rows(n, 1024, 6)
    rp, rm = oracle.adjoint(p, 0.01, w, rows=rows)
    assert e_max(gp.cpu().numpy().astype(np.float64)[rows], rp) <= TOL_POS
    assert float(np.max(np.abs(gm.cpu().numpy()[rows] - rm)) / np.max(np.abs(rm))) <= TOL_MASS


def test_calls_that_keep_the_one_sided_kernels(monkeypatch):
    cn = lib()
    torch = torch_cuda()
    n = 5000
    d, dv = dev_tensor(synth.plummer(n, 7)), dev_tensor(synth.plummer_velocities(n, 8))
    w = dev_tensor(synth.adjoint_weights(n, 9))
    one = cn.cn_force_jerk(d, dv, d.clone(), dv, 1e-3)[:2]
    both = cn.cn_force_jerk(d, dv, d, dv, 1e-3)[:2]
    adj_both = cn.cn_force_adjoint(d, 1e-3, w)
    for v in ("jerk", "adjoint"):
        cn.cn_tune_set(v, n, n, cn.cn_tune_get(v, n, n))
    try:
        tuned = cn.cn_force_jerk(d, dv, d, dv, 1e-3)[:2]
        adj_one = cn.cn_force_adjoint(d, 1e-3, w)
    finally:
        for v in ("jerk", "adjoint"):
            cn.cn_tune_set(v, n, n, None)
    assert all(torch.equal(x, y) for x, y in zip(tuned, one)) and not torch.equal(both[0], one[0])
    assert not torch.equal(adj_one[0], adj_both[0])
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        cn.cn_force_adjoint(d[:1000], 1e-3, w[:1000])
        cn.cn_force(d, d.clone(), 1e-3)
        cn.cn_force_jerk(d, dv, d.clone(), dv, 1e-3)
        cn.cn_tune_set("adjoint", n, n, cn.cn_tune_get("adjoint", n, n))
        cn.cn_force_adjoint(d, 1e-3, w)
        cn.cn_tune_set("adjoint", n, n, None)
        monkeypatch.setenv("CN_FAULT_INJECT", "capture")  # no room for the slots
        limited = cn.cn_force_jerk(d, dv, d, dv, 1e-3)[:2]
        adj_limited = cn.cn_force_adjoint(d, 1e-3, w)
        monkeypatch.delenv("CN_FAULT_INJECT")
        adj_later = cn.cn_force_adjoint(d, 1e-3, w)
        later = cn.cn_force_jerk(d, dv, d, dv, 1e-3)[:2]
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(limited, one)) and all(torch.equal(x, y) for x, y in zip(later, both))
    assert all(torch.equal(x, y) for x, y in zip(adj_limited, adj_one))
    assert all(torch.equal(x, y) for x, y in zip(adj_later, adj_both))
    assert cn.cn_get_device_status() == 0
