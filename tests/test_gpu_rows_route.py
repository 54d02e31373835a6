"""Which calls take the row kernel: those it runs faster, by the sizes and the
pair kernel's schedule of the call. A registered default shape keeps the pair
kernel, so equal bits tell the route. Every result against the FP64 oracle."""

import numpy as np
import pytest

import oracle
from gpu_common import dev_tensor, e_max, lib
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _route(call, variant, n_i, n_j):
    cn = lib()
    pi, pj = synth.plummer(n_i, 1), synth.hernquist(n_j, 2)
    pi[:, 3] = 1e-3
    di, dj = dev_tensor(pi), dev_tensor(pj)
    run = (lambda: cn.cn_force_eps_i(di, dj)) if call == "eps_i" else (lambda: cn.cn_force(di, dj, 1e-3))
    a, _ = run()
    cn.cn_tune_set(variant, n_i, n_j, cn.cn_tune_get(variant, n_i, n_j))
    try:
        pair, _ = run()
    finally:
        cn.cn_tune_set(variant, n_i, n_j, None)
    assert cn.cn_get_device_status() == 0
    rows = synth.sample_rows(n_i, 128, 3)
    ref, _ = oracle.force(pi, pj, float(np.float32(1e-3)), rows=rows, potential=False)
    assert e_max(a.cpu().numpy()[rows], ref) <= TOL
    return "pair" if bool((a == pair).all()) else "rows"


@pytest.mark.parametrize("n_i,n_j,route", [
    (135, 180000, "pair"), (145, 170003, "pair"), (300, 130000, "rows"), (401, 61003, "rows"),  # tiles filled badly, well
    (5990, 6938, "pair"), (6136, 7916, "pair"), (6750, 3592, "rows"),  # a full schedule of the pair kernel, one with gaps
    (4000, 16384, "rows"), (10007, 30011, "pair")])
def test_plain(n_i, n_j, route):
    assert _route("force", "f32", n_i, n_j) == route


@pytest.mark.parametrize("n_i,n_j,route", [
    (24000001, 1, "pair"), (800000, 31, "pair"), (750000, 33, "pair"), (150001, 200, "pair"),  # few j records
    (17999, 1343, "pair"), (6750, 3592, "rows"), (135, 180000, "pair"),
    (1400001, 31, "rows"), (220003, 200, "rows"), (16384, 16384, "rows")])
def test_per_particle_softening(n_i, n_j, route):
    assert _route("eps_i", "f32_eps_i", n_i, n_j) == route
