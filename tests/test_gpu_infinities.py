"""Results above the FP32 range come out as infinities of the right sign, as
a plain sum gives them, and not as NaN: two clumps of coincident particles, so
that every term of a component has one sign and only the particles' own masses
decide whether it overflows."""

import numpy as np
import pytest

from gpu_common import dev_tensor, lib, torch_cuda

pytestmark = pytest.mark.gpu

HEAVY = 1e38


def _clumps(n, equal, seed):
    """n particles, an eighth of them at (1, 1, 1), the others at (-1, -1, -1),
    in random order. All of them, or the first clump alone, are so heavy
    that 400 of them overflow an acceleration at that distance."""
    near = np.random.default_rng(seed).permutation(n) < n // 8
    p = np.full((n, 4), -1.0, dtype=np.float32)
    p[near, :3] = 1.0
    p[:, 3] = np.where(near | equal, HEAVY, 1e-3).astype(np.float32)
    return p, near


def _check(a, pot, near, equal):
    """First clump at +: pulled to minus infinity by the others where they are heavy."""
    a = a.cpu().numpy()
    assert np.all(np.isposinf(a[~near]))
    if equal:
        assert np.all(np.isneginf(a[near]))
    else:
        assert np.all(np.isfinite(a[near])) and np.all(a[near] < 0)
    if pot is not None:
        pot = pot.cpu().numpy()
        assert np.all(np.isneginf(pot[~near]))
        assert np.all(np.isneginf(pot[near]) if equal else np.isfinite(pot[near]))


@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("n", [4200, 13000])
def test_force_of_one_set(n, equal):
    cn = lib()
    p, near = _clumps(n, equal, n)
    d = dev_tensor(p)
    _check(*cn.cn_force(d, d, 1.0), near, equal)
    _check(*cn.cn_force(d, d, 1.0, potential=True), near, equal)
    _check(*cn.cn_force_symmetric(d, 0.0, potential=True), near, equal)
    cn.cn_tune_set("symmetric", n, n, {"i_per_thread": 4, "threads": 128, "j_tile": 128, "stages": 3, "chunk_units": 2})
    try:  # rows of tiles in bands, with sums carried from one to the next
        _check(*cn.cn_force_symmetric(d, 1.0, potential=True), near, equal)
    finally:
        cn.cn_tune_set("symmetric", n, n, None)
    plan = cn.BatchPlan(np.array([0, n], dtype=np.int64), np.ones(1, dtype=np.float32), potential=True)
    _check(*plan.run(d), near, equal)
    plan.close()
    assert cn.cn_get_device_status() == 0


@pytest.mark.parametrize("equal", [True, False])
def test_jerk_of_one_set(equal):
    cn = lib()
    n = 4200
    p, near = _clumps(n, equal, 1)
    v = np.zeros((n, 4), dtype=np.float32)
    v[near, :3] = (1.0, 2.0, 3.0)  # w - b d of a pair is (-4.5, -3.5, -2.5) for the second clump
    d, dv = dev_tensor(p), dev_tensor(v)
    a, j, pot = cn.cn_force_jerk(d, dv, d, dv, 1.0, potential=True)
    _check(a, pot, near, equal)
    assert np.all(np.isneginf(j.cpu().numpy()[~near]))
    assert cn.cn_get_device_status() == 0


@pytest.mark.parametrize("n_i,n_j", [(1000, 30011), (129, 200000), (20000, 30000)])
@pytest.mark.parametrize("equal", [True, False])
def test_one_set_on_another(n_i, n_j, equal):
    cn = lib()
    torch_cuda()
    pj, _ = _clumps(n_j, equal, 2)
    pi = np.full((n_i, 4), -1.0, dtype=np.float32)
    pi[:, 3] = 1.0
    di, dj = dev_tensor(pi), dev_tensor(pj)
    for a, pot in (cn.cn_force(di, dj, 1.0), cn.cn_force(di, dj, 1.0, potential=True), cn.cn_force_eps_i(di, dj),
                   cn.cn_force_eps_i(di, dj, potential=True)):
        _check(a, pot, np.zeros(n_i, dtype=bool), equal)
    assert cn.cn_get_device_status() == 0
