"""Terms that the kernels form without a mass (r^-3 d, and r^-3 times a
relative velocity or weight, summed and then scaled where masses are equal)
at values where they leave the FP32 range although the results, and the terms
with their masses, are well inside it: softenings far above and below the
separations with heavy and light masses, very fast and very slow particles,
very large and very small weights. Each form that takes such terms, against
the FP64 oracle.

Errors are taken in the 2-norm over the particles: in the harmonic core of a
softening far above the separations a single force cancels towards the
centre. A term carries about ten roundings and the inverse square root's
error, 1e-6 together; the sums of the terms' sizes are within a factor of
about three of the sums in that norm."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5
TOL_JERK, TOL_GRAD = 2e-5, 1.5e-5
# (length, eps2, mass): the first, the third and the fourth underflow without the mass
SETS = [(1e10, 1e32, 1e25), (1e10, 1e25, 1e20), (1e-15, 1e18, 1e34), (1e10, 9e23, 1e26)]


def _set(n, length, mass, equal, seed):
    p = synth.plummer(n, seed)
    p[:, :3] *= np.float32(length)
    p[:, 3] = np.float32(mass)
    if not equal:
        p[:, 3] *= np.random.default_rng(seed).lognormal(size=n).astype(np.float32)
    return p


def _err(x, ref):
    x = x.cpu().numpy().astype(np.float64)
    return float(np.linalg.norm(x - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("length,eps2,mass", SETS)
def test_force_forms(length, eps2, mass, equal):
    cn = lib()
    torch = torch_cuda()
    eps2 = float(np.float32(eps2))
    n = 4200
    p = _set(n, length, mass, equal, 1)
    d = dev_tensor(p)
    rows = synth.sample_rows(n, 512, 2)
    ref, rpot = oracle.force(p, p, eps2, rows=rows)
    for a, pot in (cn.cn_force(d, d, eps2), cn.cn_force(d, d, eps2, potential=True),
                   cn.cn_force_symmetric(d, eps2, potential=True)):
        assert _err(a[rows], ref) <= TOL
        if pot is not None:
            assert _err(pot[rows], rpot) <= TOL
    # an ensemble in the symmetric form: clusters large enough for it
    offs = np.array([0, 4200, 8400, 14000], dtype=np.int64)
    q = np.concatenate([_set(int(m), length, mass, equal, 3 + c) for c, m in enumerate(np.diff(offs))])
    plan = cn.BatchPlan(offs, np.full(3, eps2, dtype=np.float32))
    a, _ = plan.run(dev_tensor(q))
    plan.close()
    for lo, hi in zip(offs[:-1], offs[1:]):
        r = synth.sample_rows(int(hi - lo), 256, 4)
        ref, _ = oracle.force(q[lo:hi], q[lo:hi], eps2, rows=r, potential=False)
        assert _err(a[int(lo):int(hi)][r], ref) <= TOL
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("length,eps2,mass", SETS)
def test_one_set_on_another(length, eps2, mass, equal):
    cn = lib()
    eps2 = float(np.float32(eps2))
    pi, pj = _set(1000, length, mass, True, 5), _set(60000, length, mass, equal, 6)
    pe = pi.copy()
    pe[:, 3] = eps2
    pe[::3, 3] = np.float32(eps2 * 0.5)
    rows = synth.sample_rows(1000, 256, 7)
    ref, rpot = oracle.force(pi, pj, eps2, rows=rows)
    eref, epot = oracle.force_eps_i(pe, pj, rows=rows)
    di, dj, de = dev_tensor(pi), dev_tensor(pj), dev_tensor(pe)
    for a, pot in (cn.cn_force(di, dj, eps2), cn.cn_force(di, dj, eps2, potential=True)):
        assert _err(a[rows], ref) <= TOL
        if pot is not None:
            assert _err(pot[rows], rpot) <= TOL
    for a, pot in (cn.cn_force_eps_i(de, dj), cn.cn_force_eps_i(de, dj, potential=True)):
        assert _err(a[rows], eref) <= TOL
        if pot is not None:
            assert _err(pot[rows], epot) <= TOL
    assert cn.cn_get_device_status() == 0


# (length, eps2, mass, speed): too soft; so fast that r^-3 w overflows; so slow that it underflows
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("length,eps2,mass,speed", [(1e10, 1e32, 1e25, 1e3), (1e-9, 1e-18, 1e-30, 1e12), (1e10, 1e20, 1e30, 1e-9)])
def test_jerk(length, eps2, mass, speed, equal):
    cn = lib()
    eps2 = float(np.float32(eps2))
    n = 2100
    p = _set(n, length, mass, equal, 8)
    v = synth.plummer_velocities(n, 9) * np.float32(speed)
    rows = synth.sample_rows(n, 512, 10)
    ra, rj, rp = oracle.force_jerk(p[rows], v[rows], p, v, eps2)
    d, dv = dev_tensor(p), dev_tensor(v)
    for pot in (False, True):
        a, j, phi = cn.cn_force_jerk(d, dv, d, dv, eps2, potential=pot)
        assert _err(a[rows], ra) <= TOL
        assert _err(j[rows], rj) <= TOL_JERK
        if pot:
            assert _err(phi[rows], rp) <= TOL
    assert cn.cn_get_device_status() == 0


# (length, eps2, mass, weight): g w overflows; g w underflows
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("length,eps2,mass,weight", [(1e-6, 1e-12, 1e-30, 1e22), (1e10, 1e20, 1e20, 1e-10)])
def test_adjoint(length, eps2, mass, weight, equal):
    cn = lib()
    eps2 = float(np.float32(eps2))
    n = 2100
    p = _set(n, length, mass, equal, 11)
    w = synth.adjoint_weights(n, 12) * np.float32(weight)
    rows = synth.sample_rows(n, 512, 13)
    rp, rm = oracle.adjoint(p, eps2, w, rows=rows)
    gp, gm = cn.cn_force_adjoint(dev_tensor(p), eps2, dev_tensor(w))
    assert _err(gp[rows], rp) <= TOL_GRAD
    assert _err(gm[rows], rm) <= TOL_GRAD
    assert cn.cn_get_device_status() == 0
