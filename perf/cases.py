"""The work that users of this framework have it do, as measurable cases.

Every case is one call (for the differentiable form one forward and one
backward) through the public Python binding, on seeded particle sets shaped
like the paper's runs: Plummer spheres of equal masses, Hernquist spheres of
log-normal masses, ensembles of clusters and tree-code interaction lists.
`exact` gives the same sums in 64 bits with plain torch operations.
"""

import math

import numpy as np
import torch

import paper_astro_ph_0703100_gb300 as cn
from paper_astro_ph_0703100_gb300 import synth

DEVICE = "cuda"
SPAN = {  # the range of each size that a drawn case takes (log-uniform)
    "force": (256, 131072),
    "rows_i": (512, 32768),
    "rows_j": (2048, 262144),
    "eps_i": (512, 65536),
    "dd": (512, 65536),
    "symmetric": (4096, 131072),
    "gravity": (512, 65536),
    "jerk": (512, 65536),
    "host": (512, 131072),
}


def listed():
    return [
        # the smallest call in earnest: a 1024-body system with its potential, eps = 1/64 (launch latency counts)
        {"name": "force_n1024_pot", "call": "force", "n": 1024, "model": "plummer", "eps": 1.0 / 64.0, "potential": True},
        # the paper's smallest table entry: one force evaluation of an integrator's loop
        {"name": "force_n2048", "call": "force", "n": 2048, "model": "plummer", "eps": 0.0, "potential": False},
        # a mid-size cluster
        {"name": "force_n16384", "call": "force", "n": 16384, "model": "plummer", "eps": 0.0, "potential": False},
        # the paper's largest table entry and the headline workload
        {"name": "force_n131072", "call": "force", "n": 131072, "model": "plummer", "eps": 0.0, "potential": False},
        # one rank's rows, or a set of test particles, under a galaxy of unequal masses: i and j sets differ, ragged sizes
        {"name": "rows_10007x100003", "call": "rows", "n_i": 10007, "n_j": 100003, "model": "hernquist", "eps": 1e-3, "potential": False},
        # the compensated form on a cuspy galaxy of unequal masses with a small softening
        {"name": "dd_hernquist_n65536", "call": "dd", "n": 65536, "model": "hernquist", "eps": 1e-3, "potential": False},
        # the symmetric entry point with the potential (an energy check), an odd size
        {"name": "symmetric_n50001_pot", "call": "symmetric", "n": 50001, "model": "plummer", "eps": 0.0, "potential": True},
        # an ensemble of independent clusters of uneven sizes in one launch
        {"name": "batched_512", "call": "batched", "clusters": 512, "lo": 256, "hi": 16384, "sizes": 512, "potential": False},
        # a tree code's groups against their interaction lists (int32 indices into particles and nodes)
        {"name": "lists_indexed_512x256x4096", "call": "lists", "groups": 512, "group": 256, "entries": 4096, "indexed": True, "eps": 0.1, "potential": False},
        # a training step through the differentiable form: forward and the adjoint backward
        {"name": "gravity_step_n65536", "call": "gravity", "n": 65536, "model": "plummer", "eps": 0.1},
        # a Hermite integrator's evaluation: acceleration, jerk and potential
        {"name": "jerk_n16384_pot", "call": "jerk", "n": 16384, "model": "plummer", "eps": 1.0 / 256.0, "potential": True},
        # the host-buffer routine of a program that keeps its particles in host memory
        {"name": "host_n20000_pot", "call": "host", "n": 20000, "model": "plummer", "eps": 0.0, "potential": True},
    ]


def _log(rng, span):
    return int(round(math.exp(rng.uniform(math.log(span[0]), math.log(span[1])))))


def draw(rng):
    call = rng.choice(["force", "force", "force", "rows", "eps_i", "dd", "symmetric", "batched", "lists", "gravity", "jerk", "host"])
    pot = rng.random() < 0.35
    # eps = 0 in a case stands for the scaling runs' eps = 4 / N^(1/3)
    sphere = {"model": rng.choice(["plummer", "plummer", "hernquist"]), "eps": rng.choice([0.0, 0.0, 1e-3, 0.01, 0.1])}
    if call == "rows":
        return {"call": call, "n_i": _log(rng, SPAN["rows_i"]), "n_j": _log(rng, SPAN["rows_j"]), "potential": pot, **sphere}
    if call == "batched":
        lo = _log(rng, (64, 1024))
        return {"call": call, "clusters": _log(rng, (16, 512)), "lo": lo, "hi": lo * rng.randint(1, 16), "sizes": rng.randrange(1 << 16), "potential": pot}
    if call == "lists":
        return {"call": call, "groups": _log(rng, (32, 512)), "group": _log(rng, (24, 512)), "entries": _log(rng, (256, 8192)),
                "indexed": rng.random() < 0.5, "eps": rng.choice([1e-3, 0.01, 0.1]), "potential": pot}
    if call == "gravity":
        return {"call": call, "n": _log(rng, SPAN[call]), "model": sphere["model"], "eps": rng.choice([0.01, 0.05, 0.1])}
    if call == "jerk":
        return {"call": call, "n": _log(rng, SPAN[call]), "model": sphere["model"], "eps": rng.choice([1.0 / 256.0, 0.01, 0.1]), "potential": pot}
    return {"call": call, "n": _log(rng, SPAN[call]), "potential": pot, **sphere}


# ------------------------------------------------------------------ inputs

def _eps2(case, n):
    """The squared softening as the FP32 value that the library receives."""
    eps = case["eps"] if case["eps"] > 0.0 else synth.plummer_eps(n)
    return float(np.float32(eps * eps))


def _sphere(case, n, seed):
    return synth.plummer(n, seed) if case["model"] == "plummer" else synth.hernquist(n, seed)


def _host_inputs(case, seed):
    """The case's input arrays on the host, from the seed alone."""
    call = case["call"]
    if call == "batched":
        sizes = synth.ensemble_sizes(case["clusters"], case["sizes"], case["lo"], case["hi"])
        offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        rec = np.concatenate([synth.plummer(int(m), seed * 100003 + c) for c, m in enumerate(sizes)])
        eps2 = np.array([np.float32(synth.plummer_eps(int(m)) ** 2) for m in sizes], dtype=np.float32)
        return {"pos": rec, "offsets": offsets, "eps2": eps2}
    if call == "lists":
        groups, group, entries = case["groups"], case["group"], case["entries"]
        n = groups * group
        p = synth.plummer(n, seed)
        p = p[np.argsort(p[:, 0], kind="stable")]
        rng = np.random.Generator(np.random.PCG64(seed + 1))
        n_nodes = max(64, n // 4)
        nodes = np.empty((n_nodes, 4), dtype=np.float32)
        nodes[:, :3] = 4.0 * rng.standard_normal((n_nodes, 3))
        nodes[:, 3] = rng.uniform(1.0, 64.0, n_nodes) / n
        src = np.concatenate([p, nodes])
        # half of a list: particles around the group (a run of the order along x); half: nodes from all over
        near = entries // 2
        start = np.arange(groups, dtype=np.int64) * group + rng.integers(0, group, groups) - near // 2
        j_near = (start[:, None] + np.arange(near)[None, :]) % n
        j_far = n + rng.integers(0, n_nodes, (groups, entries - near))
        index = np.concatenate([j_near, j_far], axis=1).astype(np.int32).reshape(-1)
        return {"pos": p, "src": src, "index": index, "i_offsets": np.arange(groups + 1, dtype=np.int64) * group,
                "j_begin": np.arange(groups, dtype=np.int64) * entries, "j_count": np.full(groups, entries, dtype=np.int64)}
    if call == "rows":
        pj = _sphere(case, case["n_j"], seed)
        pi = _sphere(case, case["n_i"], seed + 1)
        return {"pos": pi, "src": pj, "eps2": _eps2(case, case["n_j"])}
    n = case["n"]
    got = {"pos": _sphere(case, n, seed), "eps2": _eps2(case, n)}
    if call == "eps_i":
        rng = np.random.Generator(np.random.PCG64(seed + 1))
        got["pos_eps"] = got["pos"].copy()
        got["pos_eps"][:, 3] = got["eps2"] * rng.uniform(0.5, 2.0, n)
    elif call == "gravity":
        got["w"] = synth.adjoint_weights(n, seed + 1)
    elif call == "jerk":
        got["vel"] = synth.plummer_velocities(n, seed + 1)
    return got


def prepare(case, seed):
    call = case["call"]
    h = _host_inputs(case, seed)
    s = {"call": call, "potential": bool(case.get("potential", False))}
    if call == "host":
        n = case["n"]
        s["eps2"] = h["eps2"]
        s["pos"] = torch.from_numpy(h["pos"]).pin_memory()
        s["acc"] = torch.empty((n, 3), dtype=torch.float32).pin_memory()
        s["pot"] = torch.empty(n, dtype=torch.float32).pin_memory() if s["potential"] else None
        return s
    for key in ("pos", "pos_eps", "src", "vel", "w"):
        if key in h:
            s[key] = torch.from_numpy(np.ascontiguousarray(h[key])).to(DEVICE)
    s["eps2"] = h.get("eps2")
    dt = torch.float64 if call == "dd" else torch.float32
    n = s["pos"].shape[0]
    if call != "gravity":
        s["acc"] = torch.empty((n, 3), dtype=dt, device=DEVICE)
        s["pot"] = torch.empty(n, dtype=dt, device=DEVICE) if s["potential"] else None
    if call == "gravity":
        s["pos"].requires_grad_(True)
    elif call == "jerk":
        s["jerk"] = torch.empty((n, 3), dtype=dt, device=DEVICE)
    elif call == "batched":
        s["plan"] = cn.BatchPlan(h["offsets"], h["eps2"], potential=s["potential"])
    elif call == "lists":
        eps2 = float(np.float32(case["eps"] ** 2))
        if case["indexed"]:
            s["plan"] = cn.ListPlan(h["i_offsets"], h["j_begin"], h["j_count"], eps2, potential=s["potential"],
                                    j_index=h["index"], n_src=h["src"].shape[0])
        else:
            s["plan"] = cn.ListPlan(h["i_offsets"], h["j_begin"], h["j_count"], eps2, potential=s["potential"])
            s["src"] = torch.from_numpy(h["src"][h["index"]]).to(DEVICE)
    return s


def run(state):
    s = state
    call = s["call"]
    if call == "force":
        out = cn.cn_force(s["pos"], s["pos"], s["eps2"], acc_out=s["acc"], pot_out=s["pot"])
    elif call == "rows":
        out = cn.cn_force(s["pos"], s["src"], s["eps2"], acc_out=s["acc"], pot_out=s["pot"])
    elif call == "eps_i":
        out = cn.cn_force_eps_i(s["pos_eps"], s["pos"], acc_out=s["acc"], pot_out=s["pot"])
    elif call == "dd":
        out = cn.cn_force_dd(s["pos"], s["pos"], s["eps2"], acc_out=s["acc"], pot_out=s["pot"])
    elif call == "symmetric":
        out = cn.cn_force_symmetric(s["pos"], s["eps2"], acc_out=s["acc"], pot_out=s["pot"])
    elif call == "batched":
        out = cn.cn_force_batched(s["plan"], s["pos"], s["acc"], s["pot"])
    elif call == "lists":
        out = cn.cn_force_lists(s["plan"], s["pos"], s["src"], s["acc"], s["pot"])
    elif call == "gravity":
        a = cn.gravity(s["pos"], s["eps2"])
        (grad,) = torch.autograd.grad(a, s["pos"], grad_outputs=s["w"])
        out = (a, grad)
    elif call == "jerk":
        out = cn.cn_force_jerk(s["pos"], s["vel"], s["pos"], s["vel"], s["eps2"], acc_out=s["acc"], jerk_out=s["jerk"], pot_out=s["pot"])
    else:
        out = cn.cn_force_host(s["pos"], s["pos"], s["eps2"], acc_out=s["acc"], pot_out=s["pot"])
    return {"out": [x for x in out if x is not None]}


def _pairs(case):
    """(ordered pairs, i-particles, j records read)."""
    call = case["call"]
    if call == "rows":
        return case["n_i"] * case["n_j"], case["n_i"], case["n_j"]
    if call == "batched":
        sizes = synth.ensemble_sizes(case["clusters"], case["sizes"], case["lo"], case["hi"]).astype(np.float64)
        return float((sizes * sizes).sum()), float(sizes.sum()), 0.0
    if call == "lists":
        n = case["groups"] * case["group"]
        src = n + max(64, n // 4) if case["indexed"] else case["groups"] * case["entries"]
        return float(n) * case["entries"], n, src + (case["groups"] * case["entries"] / 4.0 if case["indexed"] else 0.0)
    return float(case["n"]) ** 2, case["n"], 0.0


def work(case):
    """Floating-point operations of one pass (a fused multiply-add counts two;
    where the i set is the j set the terms common to a pair count once for
    both its sides) and the bytes of its inputs and outputs."""
    call = case["call"]
    pairs, ni, nj = _pairs(case)
    pot = 1.0 if case.get("potential") else 0.0
    one_sided = 19.0 + 2.0 * pot      # difference 3, softened square 6, rsqrt 1, m r^-3 3, sums 6
    shared = 13.0 + 2.0 * pot         # the same with the common half of the work done once per unordered pair
    out_b = 12.0 + 4.0 * pot
    in_b = 16.0
    if call in ("rows", "eps_i", "lists"):
        per = one_sided
    elif call == "dd":
        per, out_b = 60.0 + 6.0 * pot, 24.0 + 8.0 * pot
    elif call == "jerk":
        per, in_b, out_b = 28.0 + 2.0 * pot, 32.0, 24.0 + 4.0 * pot
    elif call == "gravity":
        per, in_b, out_b = shared + 32.0, 28.0, 28.0
    else:
        per = shared
    return {"bytes": float(ni * (in_b + out_b) + nj * 16.0), "flops": float(pairs * per)}


# ------------------------------------------------------------------ the same sums in 64 bits

def _rows_of(n_j):
    return max(1, (1 << 24) // max(1, n_j))


def _force64(pi, pj, eps2, pot):
    """a and phi of the i rows under the j records; eps2: a number or one per row."""
    acc = torch.empty((pi.shape[0], 3), dtype=torch.float64, device=pi.device)
    phi = torch.empty(pi.shape[0], dtype=torch.float64, device=pi.device)
    step = _rows_of(pj.shape[0])
    for i in range(0, pi.shape[0], step):
        d = [pj[None, :, c] - pi[i:i + step, None, c] for c in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        e = eps2 if isinstance(eps2, float) else eps2[i:i + step, None]
        r = torch.rsqrt(d2 + e)
        mr = pj[None, :, 3] * r
        q = mr * r * r
        for c in range(3):
            acc[i:i + step, c] = (q * d[c]).sum(1)
        if pot:
            phi[i:i + step] = -torch.where(d2 != 0, mr, torch.zeros_like(mr)).sum(1)
    return [acc, phi] if pot else [acc]


def _jerk64(p, v, eps2, pot):
    n = p.shape[0]
    acc, jerk = (torch.empty((n, 3), dtype=torch.float64, device=p.device) for _ in range(2))
    phi = torch.empty(n, dtype=torch.float64, device=p.device)
    step = _rows_of(n)
    for i in range(0, n, step):
        d = [p[None, :, c] - p[i:i + step, None, c] for c in range(3)]
        w = [v[None, :, c] - v[i:i + step, None, c] for c in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        r = torch.rsqrt(d2 + eps2)
        mr = p[None, :, 3] * r
        q = mr * r * r
        b = 3.0 * (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * r * r
        for c in range(3):
            acc[i:i + step, c] = (q * d[c]).sum(1)
            jerk[i:i + step, c] = (q * (w[c] - b * d[c])).sum(1)
        if pot:
            phi[i:i + step] = -torch.where(d2 != 0, mr, torch.zeros_like(mr)).sum(1)
    return [acc, jerk, phi] if pot else [acc, jerk]


def _adjoint64(p, w, eps2):
    """dL/dx and dL/dm of L = sum_i w_i . a_i, as one (n, 4) tensor."""
    n = p.shape[0]
    grad = torch.empty((n, 4), dtype=torch.float64, device=p.device)
    step = max(1, _rows_of(n) // 2)
    for k in range(0, n, step):
        rows = slice(k, k + step)
        d = [p[None, :, c] - p[rows, None, c] for c in range(3)]
        u = [p[rows, None, 3] * w[None, :, c] - p[None, :, 3] * w[rows, None, c] for c in range(3)]
        s = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2
        g = s.pow(-1.5)
        h = 3.0 * g / s * (d[0] * u[0] + d[1] * u[1] + d[2] * u[2])
        for c in range(3):
            grad[rows, c] = (g * u[c] - h * d[c]).sum(1)
        grad[rows, 3] = -(g * (w[None, :, 0] * d[0] + w[None, :, 1] * d[1] + w[None, :, 2] * d[2])).sum(1)
    return grad


def exact(case, seed):
    call = case["call"]
    pot = bool(case.get("potential", False))
    h = _host_inputs(case, seed)
    wide = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEVICE).double()  # noqa: E731
    p = wide(h["pos"])
    if call == "rows":
        out = _force64(p, wide(h["src"]), h["eps2"], pot)
    elif call == "eps_i":
        e = wide(h["pos_eps"])
        out = _force64(e, p, e[:, 3], pot)
    elif call in ("batched", "lists"):
        parts = []
        if call == "batched":
            off = h["offsets"]
            for c in range(case["clusters"]):
                x = p[off[c]:off[c + 1]]
                parts.append(_force64(x, x, float(h["eps2"][c]), pot))
        else:
            src, index = wide(h["src"]), torch.from_numpy(h["index"].astype(np.int64)).to(DEVICE)
            eps2 = float(np.float32(case["eps"] ** 2))
            for g in range(case["groups"]):
                rec = src[index[g * case["entries"]:(g + 1) * case["entries"]]]
                parts.append(_force64(p[g * case["group"]:(g + 1) * case["group"]], rec, eps2, pot))
        out = [torch.cat(x) for x in zip(*parts)]
    elif call == "gravity":
        out = [_force64(p, p, h["eps2"], False)[0], _adjoint64(p, wide(h["w"]), h["eps2"])]
    elif call == "jerk":
        out = _jerk64(p, wide(h["vel"]), h["eps2"], pot)
    else:
        out = _force64(p, p, h["eps2"], pot)
    return {"out": out}
