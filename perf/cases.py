"""Timed workloads of the library, each through its public entry points.

A case is a dict of plain values.  Its "kind" says which call it makes:

  energy_grad  System.energy_grad: E and grad E of one system
  energy       System.energy: E alone (what a scan over poses asks for)
  minimize     System.minimize, a capped run of one method on one system or a
               batch (the runs differ from a full one in their length only)
  gradfree     System.minimize with the gradient-free search, one sweep of
               moves, one atom at a time (parts = 0) or in parallel epochs
  noalloc      ffmin_pair_energy_grad_noalloc on caller-owned buffers
  train        ffmin_mlp_train: Adam steps of the preconditioner network

Inputs: chain globules of the repository's generator (0.1 atoms per cubic A,
1.5 A bonds).  A chain of a given length is grown once per process; charges,
Lennard-Jones parameters, torsions and the coordinate jitter come from the
seed.  Single evaluations take the clashing starts of the repository's
workloads (0.3 A jitter); minimizations start from a built model whose bonds
are roughly at length (0.1 A jitter), as a refinement does.

A MIXED result carries FP32 pair terms in an FP64 container: a program that
asks for that precision keeps the result in float32, and so do these cases.
"""
import functools
import math

import numpy as np
import torch

from paper_1810_03358_gb300 import ffmin, learn, synth

DEVICE = "cuda"
FP64, MIXED = ffmin.FFMIN_FP64, ffmin.FFMIN_MIXED


def listed():
    return [
        # the smallest configured system, one plain FP64 evaluation: latency
        {"name": "eg_fp64_500", "kind": "energy_grad", "n": 500, "mixed": False, "exclusions": False},
        # the paper's 10^4 variables in MIXED: what a user's own optimizer
        # calls once per step
        {"name": "eg_mixed_3334", "kind": "energy_grad", "n": 3334, "mixed": True, "exclusions": False},
        # a force field with bonded exclusions and scaled 1-4 pairs, MIXED
        {"name": "eg_mixed_excl_5000", "kind": "energy_grad", "n": 5000, "mixed": True, "exclusions": True},
        # the largest configured system, both precisions
        {"name": "eg_fp64_30000", "kind": "energy_grad", "n": 30000, "mixed": False, "exclusions": False},
        {"name": "eg_mixed_30000", "kind": "energy_grad", "n": 30000, "mixed": True, "exclusions": False},
        # L-BFGS at paper scale with FP64 terms, and on the largest system in
        # MIXED: an E + grad and three line-search trials per step
        {"name": "lbfgs_fp64_3334", "kind": "minimize", "method": "LBFGS", "n": 3334, "n_sys": 1, "steps": 10,
         "mixed": False, "learned": False},
        {"name": "lbfgs_mixed_30000", "kind": "minimize", "method": "LBFGS", "n": 30000, "n_sys": 1, "steps": 10,
         "mixed": True, "learned": False},
        # many conformations of uneven size at once, MIXED with the learned
        # diagonal: the throughput form (200 to 5,000 atoms each)
        {"name": "lbfgs_learned_batch32", "kind": "minimize", "method": "LBFGS", "n": 5000, "n_sys": 32,
         "steps": 10, "mixed": True, "learned": True},
        # the gradient-free search: a sweep one atom at a time, and a sweep
        # in parallel epochs
        {"name": "gradfree_fp64_500", "kind": "gradfree", "n": 500, "parts": 0},
        {"name": "gradfree_epochs_3334", "kind": "gradfree", "n": 3334, "parts": 64},
        # non-bonded terms for a caller that allows no allocation
        {"name": "noalloc_fp64_4000", "kind": "noalloc", "n": 4000},
        # training of the preconditioner network on recorded samples
        {"name": "train_16384", "kind": "train", "rows": 1000000, "batch": 16384, "steps": 50},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy_grad", "energy_grad", "energy_grad", "energy", "minimize", "minimize", "gradfree",
                       "noalloc", "train"])
    if kind == "energy_grad":
        return {"kind": kind, "n": _log_int(rng, 64, 30000), "mixed": rng.random() < 0.5,
                "exclusions": rng.random() < 0.25}
    if kind == "energy":
        return {"kind": kind, "n": _log_int(rng, 64, 30000), "mixed": rng.random() < 0.5}
    if kind == "minimize":
        if rng.random() < 0.3:  # a batch of uneven sizes up to n atoms
            return {"kind": kind, "method": "LBFGS", "n": _log_int(rng, 400, 5000), "n_sys": rng.randint(2, 40),
                    "steps": rng.randint(5, 12), "mixed": True, "learned": rng.random() < 0.5}
        mixed = rng.random() < 0.5
        return {"kind": kind, "method": rng.choice(["LBFGS", "LBFGS", "CG", "GD"]),
                "n": _log_int(rng, 200, 12000 if mixed else 5000), "n_sys": 1, "steps": rng.randint(5, 12),
                "mixed": mixed, "learned": False}
    if kind == "gradfree":
        if rng.random() < 0.5:
            return {"kind": kind, "n": _log_int(rng, 100, 1200), "parts": 0}
        return {"kind": kind, "n": _log_int(rng, 500, 5000), "parts": rng.randint(4, 64)}
    if kind == "noalloc":
        return {"kind": kind, "n": _log_int(rng, 50, 8192)}
    return {"kind": kind, "rows": _log_int(rng, 20000, 4000000), "batch": _log_int(rng, 512, 32768),
            "steps": rng.randint(10, 80)}


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=256)
def _chain(n, seed):
    """Reference chain of n atoms: coordinates and bond angles (read-only)."""
    while True:
        try:
            x, theta, _ = synth.grow_chain(n, np.random.default_rng(seed))
            return x, theta
        except RuntimeError:  # growth gave up: another chain
            seed += 1000003


def _system(n, chain_seed, rng, jitter, exclusions=False):
    x_ref, theta = _chain(n, chain_seed)
    q = rng.uniform(-0.8, 0.8, size=n)
    nb, na, nd = max(n - 1, 0), max(n - 2, 0), max(n - 3, 0)
    return synth.System(
        x=np.ascontiguousarray(x_ref + rng.normal(0.0, jitter, size=x_ref.shape)), x_ref=x_ref,
        charge=q - q.mean(), sigma=rng.uniform(2.5, 3.8, size=n), epsilon=rng.uniform(0.02, 0.2, size=n),
        bond_idx=np.stack([np.arange(nb) + i for i in range(2)], axis=1).astype(np.int32),
        bond_k=np.full(nb, synth.BOND_K), bond_r0=np.full(nb, synth.BOND_LENGTH),
        angle_idx=np.stack([np.arange(na) + i for i in range(3)], axis=1).astype(np.int32),
        angle_k=np.full(na, synth.ANGLE_K), angle_theta0=theta[:na],
        dihedral_idx=np.stack([np.arange(nd) + i for i in range(4)], axis=1).astype(np.int32),
        dihedral_v=rng.uniform(0.0, 1.0, size=(nd, 4)), exclusions=1 if exclusions else 0)


def _sizes(case):
    if case.get("n_sys", 1) == 1:
        return [case["n"]]
    return [int(v) for v in synth.batch_sizes(case["n_sys"], 7, 200, case["n"])]


def _systems(case, seed):
    rng = np.random.default_rng(seed)
    jitter = 0.1 if case["kind"] in ("minimize", "gradfree") else synth.JITTER_SIGMA
    return [_system(n, 1000 + b, rng, jitter, case.get("exclusions", False)) for b, n in enumerate(_sizes(case))]


def _device(a, dtype=torch.float64):
    return torch.tensor(np.ascontiguousarray(a).reshape(-1), dtype=dtype, device=DEVICE)


def _samples(case, seed):
    """Training rows with the features' ranges in recorded trajectories."""
    rng = np.random.default_rng(seed)
    n = case["rows"]
    feat = np.empty((n, 5), dtype=np.float32)
    feat[:, 0] = rng.uniform(-0.8, 0.8, size=n)
    feat[:, 1] = rng.uniform(2.5, 3.8, size=n)
    feat[:, 2] = rng.uniform(0.02, 0.2, size=n)
    feat[:, 3] = rng.integers(20, 260, size=n) / 64.0
    feat[:, 4] = rng.gamma(3.0, 1.5, size=n)
    target = (0.4 * feat[:, 1] - 0.1 * feat[:, 4] + rng.normal(0.0, 1.4, size=n)).astype(np.float32)
    return feat, target, learn.init_weights(seed % 1000003)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        feat, target, w0 = _samples(case, seed)
        return {"case": case, "seed": seed, "feat": torch.tensor(feat, device=DEVICE), "target": _device(target, torch.float32),
                "w0": _device(w0, torch.float32), "w": _device(w0, torch.float32),
                "adam": torch.zeros(2 * learn.N_PARAMS, dtype=torch.float32, device=DEVICE),
                "work": torch.zeros(ffmin.ffmin_mlp_work_floats(), dtype=torch.float32, device=DEVICE)}
    systems = _systems(case, seed)
    x = _device(np.concatenate([s.x.reshape(-1) for s in systems]))
    if kind == "noalloc":
        s = systems[0]
        return {"case": case, "x": x, "q": _device(s.charge), "sigma": _device(s.sigma), "eps": _device(s.epsilon),
                "g": torch.empty_like(x), "e": torch.empty(1, dtype=torch.float64, device=DEVICE)}
    S = ffmin.System(systems, MIXED if case.get("mixed") else FP64)
    if case.get("learned"):
        ffmin.ffmin_set_precond(S.handle, learn.load_weights())
    return {"case": case, "S": S, "x": x, "g": torch.empty_like(x), "work": torch.empty_like(x), "seed": seed}


# ---------------------------------------------------------------- one pass
def _kept(case, v):
    """The result in the precision it has: float32 for MIXED pair terms."""
    if isinstance(v, torch.Tensor):
        return v.float() if case.get("mixed") else v
    return np.asarray(v, dtype=np.float32 if case.get("mixed") else np.float64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "energy_grad":
        e, g = state["S"].energy_grad(state["x"], state["g"])
        return {"e": _kept(case, e), "g": _kept(case, g)}
    if kind == "energy":
        return {"e": _kept(case, state["S"].energy(state["x"]))}
    if kind in ("minimize", "gradfree"):
        x = state["work"]
        x.copy_(state["x"])
        if kind == "minimize":
            res = state["S"].minimize(x, method=case["method"], max_iter=case["steps"],
                                      use_learned_precond=1 if case["learned"] else 0)
        else:
            res = state["S"].minimize(x, method="GRADFREE", max_iter=case["n"], gradfree_parts=case["parts"],
                                      seed=state["seed"])
        return {"x": _kept(case, x), "e": _kept(case, [r["energy"] for r in res]),
                "iterations": np.array([r["iterations"] for r in res], dtype=np.int64)}
    if kind == "noalloc":
        ffmin.ffmin_pair_energy_grad_noalloc(state["x"], state["q"], state["sigma"], state["eps"], state["g"],
                                             state["e"])
        return {"e": state["e"], "g": state["g"]}
    state["w"].copy_(state["w0"])
    state["adam"].zero_()
    losses = ffmin.ffmin_mlp_train(state["feat"], state["target"], case["steps"], case["batch"], 3e-3, state["seed"],
                                   state["w"], state["adam"], state["work"])
    return {"w": state["w"], "losses": losses}


def work(case):
    """Unique pairs at 35 flops (E + grad) or 23 (E); the network at 2 flops
    per weight forward and 4 backward."""
    kind = case["kind"]
    if kind == "train":
        return {"bytes": case["steps"] * (24.0 * case["batch"] + 4.0 * 7 * learn.N_PARAMS),
                "flops": 6.0 * learn.N_PARAMS * case["steps"] * case["batch"]}
    n = np.array(_sizes(case), dtype=np.float64)
    pairs, atoms = float((n * (n - 1) / 2).sum()), float(n.sum())
    if kind == "energy":
        return {"bytes": 48.0 * atoms, "flops": 23.0 * pairs}
    if kind == "minimize":
        return {"bytes": 72.0 * atoms, "flops": ((case["steps"] + 1) * 35.0 + 3.0 * case["steps"] * 23.0) * pairs}
    if kind == "gradfree":
        return {"bytes": 72.0 * atoms, "flops": 35.0 * pairs + 8.0 * 23.0 * atoms * (atoms - 1)}
    return {"bytes": 72.0 * atoms, "flops": 35.0 * pairs}


# ---------------------------------------------------------------- in 64 bits
def _exact_pairs(s, x, scales):
    """Sum over pairs, row blocks of a 64-bit all-pairs table; scales: (i, j,
    s_ij) of the pairs that count with another weight than one."""
    c = s.coulomb_c if s.coulomb_c > 0 else synth.COULOMB_KCAL
    q, sg, ep = (torch.tensor(a, dtype=torch.float64, device=DEVICE) for a in (s.charge, s.sigma, s.epsilon))
    n, e, g = x.shape[0], 0.0, torch.zeros_like(x)
    step = max(1, 20000000 // n)
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        d = x[None, :, :] - x[i0:i1, None, :]
        r2 = (d * d).sum(-1)
        own = torch.arange(i0, i1, device=DEVICE)
        r2[own - i0, own] = 1.0
        wt = torch.ones_like(r2)
        wt[own - i0, own] = 0.0
        if scales is not None:
            a, b, v = scales
            m = (a >= i0) & (a < i1)
            wt[a[m] - i0, b[m]] = v[m]
        r = r2.sqrt()
        ec = c * q[i0:i1, None] * q[None, :] / r
        s6 = (sg[i0:i1, None] * sg[None, :] / r2) ** 3
        e4 = 4.0 * (ep[i0:i1, None] * ep[None, :]).sqrt()
        e = e + 0.5 * (wt * (ec + e4 * (s6 * s6 - s6))).sum()
        f = wt * (ec + e4 * (12.0 * s6 * s6 - 6.0 * s6)) / r2
        g[i0:i1] = (f[:, :, None] * d).sum(1)
    return e, g


def _exact_bonded(s, x):
    """Bonds, angles and four-term torsions and their gradient (autograd)."""
    y = x.clone().requires_grad_(True)

    def t(a):
        return torch.tensor(a, dtype=torch.float64, device=DEVICE)

    def at(idx, k):
        return y[torch.tensor(idx[:, k], dtype=torch.long, device=DEVICE)]

    e = y.sum() * 0.0
    if len(s.bond_k):
        e = e + (t(s.bond_k) * ((at(s.bond_idx, 0) - at(s.bond_idx, 1)).norm(dim=1) - t(s.bond_r0)) ** 2).sum()
    if len(s.angle_k):
        u, v = at(s.angle_idx, 0) - at(s.angle_idx, 1), at(s.angle_idx, 2) - at(s.angle_idx, 1)
        th = torch.atan2(torch.linalg.cross(u, v).norm(dim=1), (u * v).sum(1))
        e = e + (t(s.angle_k) * (th - t(s.angle_theta0)) ** 2).sum()
    if len(s.dihedral_v):
        p = [at(s.dihedral_idx, k) for k in range(4)]
        b1, b2, b3 = p[1] - p[0], p[2] - p[1], p[3] - p[2]
        m, n = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
        phi = torch.atan2(b2.norm(dim=1) * (b1 * n).sum(1), (m * n).sum(1))
        v = t(s.dihedral_v)
        e = e + 0.5 * (v[:, 0] * (1 + phi.cos()) + v[:, 1] * (1 - (2 * phi).cos()) + v[:, 2] * (1 + (3 * phi).cos())
                       + v[:, 3] * (1 - (4 * phi).cos())).sum()
    e.backward()
    return e.detach(), y.grad


def _exact_scales(s):
    scale = {}
    for idx, v in ((s.bond_idx, 0.0), (s.angle_idx, 0.0), (s.dihedral_idx, s.scale14)):
        for row in idx:
            i, j = int(row[0]), int(row[-1])
            for k in ((i, j), (j, i)):
                scale[k] = min(scale.get(k, 1.0), v)
    ij = torch.tensor(list(scale), dtype=torch.long, device=DEVICE)
    return ij[:, 0], ij[:, 1], torch.tensor(list(scale.values()), dtype=torch.float64, device=DEVICE)


def _mulhi(a, b):
    """High 64 bits of a 64 x 64-bit product (numpy uint64)."""
    m, k = np.uint64(0xFFFFFFFF), np.uint64(32)
    al, ah, bl, bh = a & m, a >> k, b & m, b >> k
    mid = ah * bl + ((al * bl) >> k)
    return ah * bh + (mid >> k) + ((al * bh + (mid & m)) >> k)


def _exact_train(case, seed):
    feat, target, w0 = _samples(case, seed)
    rows, batch = case["rows"], case["batch"]
    f = torch.tensor(feat, dtype=torch.float64, device=DEVICE)
    t = torch.tensor(target, dtype=torch.float64, device=DEVICE)
    w = torch.tensor(w0, dtype=torch.float64, device=DEVICE)
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
    with np.errstate(over="ignore"):
        for step in range(case["steps"]):
            k = np.arange(batch, dtype=np.uint64) + np.uint64(step * batch + 1)
            z = np.uint64(seed) + k * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
            row = torch.tensor(_mulhi(z, np.uint64(rows)).astype(np.int64), device=DEVICE)
            y = w.clone().requires_grad_(True)
            h = torch.relu(f[row] @ y[:320].view(64, 5).T + y[320:384])
            loss = ((h @ y[384:448] + y[448] - t[row]) ** 2).mean()
            loss.backward()
            m, v = 0.9 * m + 0.1 * y.grad, 0.999 * v + 0.001 * y.grad ** 2
            w = w - 3e-3 * (m / (1 - 0.9 ** (step + 1))) / ((v / (1 - 0.999 ** (step + 1))).sqrt() + 1e-8)
            losses.append(float(loss.detach()))
    return {"w": w, "losses": np.array(losses)}


def exact(case, seed):
    """E and grad E from their definitions, the training run step by step.
    The minimizers' trajectories have no such value: each step's point
    follows from the rounding of all steps before it."""
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind not in ("energy_grad", "energy", "noalloc"):
        return None
    s = _systems(case, seed)[0]
    x = _device(s.x).view(-1, 3)
    e, g = _exact_pairs(s, x, _exact_scales(s) if s.exclusions else None)
    if kind != "noalloc":
        eb, gb = _exact_bonded(s, x)
        e, g = e + eb, g + gb
    e = e.reshape(1)
    return {"e": e} if kind == "energy" else {"e": e, "g": g.reshape(-1)}
