"""The native marshalling of cn_force, cn_force_dd and cn_force_eps_i: results
equal to the Python one's bit for bit over every form of the outputs, streams
and empty sets; and whatever it does not take is handled or refused as there."""

import numpy as np
import pytest

from gpu_common import dev_tensor, lib, torch_cuda
from paper_astro_ph_0703100_gb300 import synth

pytestmark = pytest.mark.gpu


def _both(cn, call):
    """call() with and without the native marshalling."""
    native = cn._load_native()
    assert native is not False
    seen = []

    class Spy:
        rows = native.rows

        @staticmethod
        def force(*a):
            seen.append(native.force(*a))
            return seen[-1]

        @staticmethod
        def force_eps_i(*a):
            seen.append(native.force_eps_i(*a))
            return seen[-1]

    def result():
        try:
            out = call()
        except Exception as e:  # the same refusal on both paths
            return type(e), str(e)
        torch_cuda().cuda.synchronize()
        return tuple(x.clone() if x is not None else None for x in out)

    cn._native = Spy
    try:
        a = result()
        cn._native = False
        b = result()
    finally:
        cn._native = native
    return a, b, seen


def _same(a, b):
    torch = torch_cuda()
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert torch.equal(x, y) if isinstance(x, torch.Tensor) else x == y


@pytest.mark.parametrize("n_i,n_j", [(1, 1), (100, 3), (0, 5), (5, 0), (2048, 2048), (5000, 5003)])
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("pot", [False, True])
def test_same_as_python(n_i, n_j, given, pot):
    cn = lib()
    torch = torch_cuda()
    pi, pj = dev_tensor(synth.plummer(max(n_i, 1), 1))[:n_i], dev_tensor(synth.plummer(max(n_j, 1), 2))[:n_j]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for name, dt in (("cn_force", torch.float32), ("cn_force_dd", torch.float64), ("cn_force_eps_i", torch.float32)):
        fn = getattr(cn, name)
        args = (pi, pj) if name == "cn_force_eps_i" else (pi, pj, 1e-3)
        out = dict(acc_out=torch.empty((n_i, 3), dtype=dt, device="cuda"),
                   pot_out=torch.empty((n_i,), dtype=dt, device="cuda") if pot else None) if given else dict(potential=pot)
        a, b, seen = _both(cn, lambda: fn(*args, **out))
        assert seen == [0]
        _same(a, b)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            here, _, seen = _both(cn, lambda: fn(*args, **out))
        there, _, _ = _both(cn, lambda: fn(*args, **out, stream=s))
        torch.cuda.synchronize()
        assert seen == [0]
        _same(a, here)
        _same(a, there)


def test_refusals_are_the_python_ones():
    cn = lib()
    torch = torch_cuda()
    p = dev_tensor(synth.plummer(64, 3))
    acc = torch.empty((64, 3), device="cuda")
    calls = [
        lambda: cn.cn_force(p.cpu(), p, 1e-3),
        lambda: cn.cn_force(p.double(), p, 1e-3),
        lambda: cn.cn_force(p, p[:, :3], 1e-3),
        lambda: cn.cn_force(p.t().contiguous().t(), p, 1e-3),
        lambda: cn.cn_force(p.cpu().numpy(), p, 1e-3),
        lambda: cn.cn_force(p, p, 1e-3, acc_out=acc[:63]),
        lambda: cn.cn_force(p, p, 1e-3, acc_out=acc.double()),
        lambda: cn.cn_force(p, p, 1e-3, acc_out=acc, pot_out=acc),
        lambda: cn.cn_force(p, p, -1.0, acc_out=acc),
        lambda: cn.cn_force(p, p, float("nan"), acc_out=acc),
        lambda: cn.cn_force(p, p, None, acc_out=acc),
        lambda: cn.cn_force(p, p, 1e-3, acc_out=p.view(-1)[:192].view(64, 3)),
        lambda: cn.cn_force(p.view(-1)[1:-3].view(63, 4), p, 1e-3),  # misaligned records
    ]
    for k, call in enumerate(calls):
        a, b, seen = _both(cn, call)
        assert a == b and isinstance(a[0], type), (k, a, b)
        assert 0 not in seen, k


def test_what_python_takes_too():
    cn = lib()
    torch = torch_cuda()
    p = dev_tensor(synth.plummer(64, 3))

    class Sub(torch.Tensor):
        pass

    for eps2 in (1, np.float32(1e-3), np.float64(1e-3), torch.tensor(1e-3), "1e-3"):
        a, b, _ = _both(cn, lambda: cn.cn_force(p, p, eps2, potential=True))
        _same(a, b)
    for q in (torch.nn.Parameter(p), p.clone().requires_grad_(True), p.as_subclass(Sub), p[:0], p[3:]):
        a, b, _ = _both(cn, lambda: cn.cn_force(q, p, 1e-3, potential=True))
        _same(a, b)
