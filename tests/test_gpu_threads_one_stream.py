"""Calls of several host threads on one stream, whose workspace has its size
already: each call's result is that of the same call alone, also for the forms
that take more than one launch."""

import threading

import numpy as np
import pytest

from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu

THREADS, CALLS = 4, 150


def _calls(cn, form, seed):
    """The inputs of one thread and its call: outputs as a tuple of tensors."""
    n = 1500 if form == "adjoint_small" else 5000
    d = dev_tensor(synth.hernquist(n, seed))
    if form == "force":
        return lambda: (cn.cn_force(d, d, 1e-3)[0],)
    if form == "symmetric":
        return lambda: (cn.cn_force_symmetric(d, 1e-3)[0],)
    if form == "rows":
        j = dev_tensor(synth.hernquist(40000, 50 + seed))
        i = d[:1000].contiguous()
        return lambda: (cn.cn_force(i, j, 1e-3)[0],)
    if form == "eps_i":
        e = d.clone()
        e[:, 3] = 1e-3
        return lambda: (cn.cn_force_eps_i(e, d)[0],)
    if form == "jerk":
        v = dev_tensor(synth.plummer_velocities(n, seed))
        return lambda: cn.cn_force_jerk(d, v, d, v, 1e-3)[:2]
    if form.startswith("adjoint"):
        w = dev_tensor(synth.adjoint_weights(n, seed))
        return lambda: cn.cn_force_adjoint(d, 1e-3, w)
    offs = np.array([0, 2000, 5000], dtype=np.int64)
    plan = cn.BatchPlan(offs, np.full(2, 1e-3, dtype=np.float32))
    return lambda: (plan.run(d)[0],)


@pytest.mark.parametrize("form", ["force", "symmetric", "rows", "eps_i", "jerk", "adjoint", "adjoint_small", "ensemble"])
def test_each_call_as_alone(form):
    cn = lib()
    torch = torch_cuda()
    calls = [_calls(cn, form, 1 + t) for t in range(THREADS)]
    alone = [c() for c in calls]
    torch.cuda.synchronize()
    out = [[] for _ in calls]
    start = threading.Barrier(THREADS)

    def work(t):
        start.wait()
        for _ in range(CALLS):
            out[t].append(calls[t]())

    threads = [threading.Thread(target=work, args=(t,)) for t in range(THREADS)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert cn.cn_get_device_status() == 0
    wrong = sum(not torch.equal(x, y) for t in range(THREADS) for got in out[t] for x, y in zip(got, alone[t]))
    assert all(len(o) == CALLS for o in out) and wrong == 0
