"""Performance cases: what a user of this framework has it do, through its public calls.

listed() names the cases, draw() makes more of the same ranges, prepare() builds
what a program holds before the call (a population, a model, device arrays),
run() is one pass, work() its unavoidable bytes and operations and exact() the
same results from plain torch or numpy in 64 bits where they are defined
without the framework.

Kinds (each case has a "kind"):
  anneal     a whole population anneal, pamd_reset + pamd_anneal: the product.
             The MD is chaotic, so its averages have no 64-bit value of their own.
  batch      the same for many molecules of uneven size in one context.
  fp64       the all-FP64 mode: one propagate block and the state it leaves.
  resample   resampling of a large population with its gather: one cooling and
             one heating step, so that repeated passes keep the temperature,
             and the averages of the gathered population.
  label      exact forces and energies of given configurations (training labels).
  energy     surrogate energies and forces, or energies and their autograd gradient.
  train      minibatch steps of the surrogate's force-matching training.
  normalize  feature and energy statistics of a training set.
  drive      a propagate block driven by the surrogate.
  wham       multiple-histogram reweighting of recorded energies.

Positions, velocities and forces of the mixed-precision calls are FP32 values
(the binding widens them); they are kept as FP32 here, as a training set or a
trajectory file keeps them.
"""
import math

import numpy as np
import torch

import pamd_inputs as pi
from paper_1806_06016_gb300 import pamd
from paper_1806_06016_gb300 import surrogate

KB = 0.008314462618
KE = 138.935458
DT = 0.001
# thermal displacement per coordinate (nm): a bond of the chain at about 600 K and, for the surrogate, 1500 K
JITTER_COLD, JITTER = 0.005, 0.008


def listed():
    return [
        # the smallest anneal in use: 22 atoms, 256 replicas, 20 temperature steps; latency and launches count
        {"name": "anneal_22x256", "kind": "anneal", "atoms": 22, "replicas": 256, "steps": 20, "theta": 100,
         "t_first": 1000.0, "t_last": 300.0, "rule": 0, "resample": True, "chain": True},
        # the benchmark's population (75 atoms, 8192 replicas, theta = 1000), the first steps of its schedule
        {"name": "anneal_75x8192", "kind": "anneal", "atoms": 75, "replicas": 8192, "steps": 2, "theta": 1000,
         "t_first": 1000.0, "t_last": 972.7, "rule": 0, "resample": True, "chain": True},
        # the batched workload's 16 molecules of 20..200 atoms, 4096 replicas each, shorter blocks
        {"name": "batch_16x4096", "kind": "batch", "molecules": 16, "replicas": 4096, "steps": 2, "theta": 100,
         "t_first": 800.0, "t_last": 769.2},
        # the precision study's population in the all-FP64 mode
        {"name": "fp64_75x2048", "kind": "fp64", "atoms": 75, "replicas": 2048, "theta": 20, "chain": True},
        # resampling of the largest population in use: weights, scans, copy counts, gather of 2 x 1.9 GB
        {"name": "resample_75x1048576", "kind": "resample", "atoms": 75, "replicas": 1 << 20, "rule": 0},
        # labelling a recorded population with exact forces, as each step of a harvest does
        {"name": "label_75x8192", "kind": "label", "atoms": 75, "replicas": 8192, "chain": True},
        # a small differentiable surrogate call: energies and their gradient
        {"name": "energy_22x256", "kind": "energy", "atoms": 22, "hidden": 128, "samples": 256, "autograd": True},
        # surrogate energies and forces of a whole population
        {"name": "energy_75x65536", "kind": "energy", "atoms": 75, "hidden": 512, "samples": 65536, "autograd": False},
        # training at the benchmark's minibatch of 2048
        {"name": "train_75x2048", "kind": "train", "atoms": 75, "hidden": 512, "batch": 2048, "minibatches": 4},
        # normalisation of a training set before training starts
        {"name": "normalize_75x65536", "kind": "normalize", "atoms": 75, "hidden": 512, "samples": 65536},
        # a surrogate-driven block
        {"name": "drive_75x16384", "kind": "drive", "atoms": 75, "hidden": 512, "replicas": 16384, "theta": 20},
        # reweighting of the benchmark anneal's energies (101 temperatures, 8192 replicas, 2000 bins)
        {"name": "wham_101x8192", "kind": "wham", "temps": 101, "replicas": 8192, "bins": 2000, "sweeps": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anneal", "batch", "fp64", "resample", "label", "energy", "train", "normalize", "drive", "wham"])
    c = {"kind": kind}
    if kind == "anneal":
        n, r = _log(rng, 10, 200), _log(rng, 64, 8192)
        # at most about the benchmark population's three blocks of 1000 steps
        budget = 75 * 75 * 8192 * 1000
        theta = rng.choice([20, 50, 100, 200, 500])
        steps = rng.randint(1, 20)
        while theta > 20 and n * n * r * theta * (steps + 1) > budget:
            theta //= 2
        while steps > 1 and n * n * r * theta * (steps + 1) > budget:
            steps -= 1
        c.update(atoms=n, replicas=r, steps=steps, theta=theta, t_first=1000.0,
                 t_last=1000.0 * (0.985 ** steps), rule=rng.choice([0, 0, 1]), resample=rng.random() < 0.8,
                 chain=rng.random() < 0.8)
    elif kind == "batch":
        c.update(molecules=rng.randint(2, 16), replicas=_log(rng, 128, 2048), steps=rng.randint(1, 3),
                 theta=rng.choice([20, 50, 100]), t_first=800.0, t_last=784.0)
    elif kind == "fp64":
        n = _log(rng, 10, 128)
        c.update(atoms=n, replicas=_log(rng, 64, max(64, min(4096, 75 * 75 * 2048 // (n * n)))),
                 theta=rng.randint(5, 20), chain=rng.random() < 0.7)
    elif kind == "resample":
        c.update(atoms=_log(rng, 10, 100), replicas=_log(rng, 1000, 1 << 20), rule=rng.choice([0, 1]))
        c["replicas"] = min(c["replicas"], (75 << 20) // c["atoms"])
    elif kind == "label":
        n = _log(rng, 10, 200)
        c.update(atoms=n, replicas=min(_log(rng, 64, 16384), 75 * 8192 // n), chain=rng.random() < 0.8)
    elif kind == "energy":
        n = rng.choice([9, 22, 47, 75, 120, 150])
        m = min(_log(rng, 16, 65536), 65536 * 75 * 75 // (n * n))
        c.update(atoms=n, hidden=rng.choice([64, 128, 256, 512]), samples=m, autograd=rng.random() < 0.3)
    elif kind == "train":
        c.update(atoms=rng.choice([9, 22, 47, 75]), hidden=rng.choice([64, 128, 256, 512]),
                 batch=4 * _log(rng, 64, 1024), minibatches=rng.randint(1, 4))
    elif kind == "normalize":
        c.update(atoms=rng.choice([9, 22, 47, 75]), hidden=128, samples=_log(rng, 100, 65536))
    elif kind == "drive":
        n = rng.choice([22, 47, 75])
        c.update(atoms=n, hidden=rng.choice([128, 256, 512]), replicas=_log(rng, 256, 16384), theta=rng.randint(5, 20))
    else:
        nt = _log(rng, 8, 101)
        c.update(temps=nt, replicas=min(_log(rng, 256, 131072), (1 << 22) // nt), bins=_log(rng, 50, 5000),
                 sweeps=rng.randint(10, 100))
    return c


# ------------------------------------------------------------------ inputs

def _topology(case):
    top = pi.make_chain(case["atoms"], 1)
    if case.get("chain", True):
        return top
    # the same molecule with its atoms listed in another order: the general bonded path
    n = top.n_atoms
    new = np.random.default_rng(5).permutation(n).astype(np.int32)  # new index of old atom i
    old = np.argsort(new)
    for k in ("mass", "charge", "sigma", "epsilon", "x0"):
        setattr(top, k, getattr(top, k)[old])
    for k in ("bond", "angle", "dihedral", "excl", "pair14"):
        setattr(top, k, new[getattr(top, k)])
    return top


def _configurations(top, n, scale, seed):
    """[n, N, 3] float32-representable positions: the start geometry with thermal jitter."""
    return pi.perturbed_positions(top, n, scale, seed).astype(np.float32).astype(np.float64)


def _velocities(top, n, T, seed):
    v = pi.gaussian_velocities(n, top.n_atoms, 1.0, seed + 1) * np.sqrt(KB * T / top.mass)[None, :, None]
    return v.astype(np.float32).astype(np.float64)


def _device_configurations(top, n, scale, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, top.n_atoms, 3), generator=g, device="cuda") * scale
    return (x + torch.tensor(top.x0, dtype=torch.float32, device="cuda")).contiguous()


def _pairs(n):
    return torch.triu_indices(n, n, 1, device="cuda")


def _features64(x):
    i, j = _pairs(x.shape[1])
    return 1.0 / torch.linalg.vector_norm(x[:, i] - x[:, j], dim=-1)


def _network(case, seed):
    """Weights, normalisation and energy scale of a surrogate (float32 numpy arrays, as set_params takes)."""
    n, h = case["atoms"], case["hidden"]
    p = n * (n - 1) // 2
    rng = np.random.default_rng(1000 + seed)
    w = {"W1": rng.normal(0, 1 / math.sqrt(p), (h, p)), "b1": rng.normal(0, 0.1, h),
         "W2": rng.normal(0, 1 / math.sqrt(h), (h, h)), "b2": rng.normal(0, 0.1, h),
         "w3": rng.normal(0, 1 / math.sqrt(h), h)}
    w = {k: v.astype(np.float32) for k, v in w.items()}
    top = pi.make_chain(n, 1)
    g = _features64(_device_configurations(top, 512, JITTER, 77).double())
    w["mu"] = g.mean(0).cpu().numpy().astype(np.float32)
    w["sd"] = (g.std(0) + 0.05).cpu().numpy().astype(np.float32)
    w["b3"], w["mu_E"], w["sigma_E"] = 0.125, -300.0, 360.0
    return w


def _labels(n, atoms, seed):
    """Energies and forces of the size a 75-atom chain has."""
    g = torch.Generator(device="cuda").manual_seed(seed + 9)
    E = -300.0 + 360.0 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    F = 900.0 * torch.randn((n, atoms, 3), generator=g, device="cuda")
    return E, F


def _recorded(case, seed):
    """Energies [temps][replicas] with the spread of a chain's canonical distributions."""
    T = pi.geometric_schedule(1000.0, 250.0, case["temps"] - 1)
    rng = np.random.default_rng(seed)
    return T, np.stack([rng.gamma(107.0, KB * t, case["replicas"]) for t in T])


class _Batch:
    """A batch context that is freed with its owner."""

    def __init__(self, tops, replicas, T0, seed):
        n = len(tops)
        self.ctx = pamd.pamd_init_batch(tops, [replicas] * n, [T0] * n, seed, pamd.torch_options())

    def __del__(self):
        pamd.pamd_destroy(self.ctx)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed}
    if kind == "anneal":
        s["temps"] = pi.geometric_schedule(case["t_first"], case["t_last"], case["steps"])
        s["pop"] = pamd.Population(_topology(case), case["replicas"], case["t_first"], seed,
                                   pamd.torch_options(resample_rule=case["rule"]))
    elif kind == "batch":
        s["temps"] = pi.geometric_schedule(case["t_first"], case["t_last"], case["steps"])
        sizes = pi.batched_chain_sizes(case["molecules"])
        s["batch"] = _Batch([pi.make_chain(n, 1 + m) for m, n in enumerate(sizes)], case["replicas"],
                            case["t_first"], seed)
    elif kind == "fp64":
        top = _topology(case)
        s["pop"] = pamd.Population(top, case["replicas"], 600.0, seed,
                                   pamd.torch_options(precision=pamd.PAMD_PREC_FP64))
        s["pop"].set_state(_configurations(top, case["replicas"], JITTER_COLD, seed),
                           _velocities(top, case["replicas"], 600.0, seed))
    elif kind == "resample":
        s["pop"] = pamd.Population(_topology(case), case["replicas"], 1000.0, seed,
                                   pamd.torch_options(resample_rule=case["rule"]))
        s["pop"].propagate(20, DT, 1000.0)
    elif kind == "label":
        top = _topology(case)
        s["pop"] = pamd.Population(top, case["replicas"], 600.0, seed, pamd.torch_options())
        s["x"] = _configurations(top, case["replicas"], JITTER_COLD, seed)
        s["v"] = np.zeros_like(s["x"])
    elif kind in ("energy", "train", "normalize", "drive"):
        top = pi.make_chain(case["atoms"], 1)
        s["model"] = surrogate.MLP(case["atoms"], case["hidden"], seed % 1000)
        if kind != "normalize":
            s["model"].set_params(_network(case, seed))
        if kind == "energy":
            s["x"] = _device_configurations(top, case["samples"], JITTER, seed)
            s["gE"] = torch.ones(case["samples"], dtype=torch.float64, device="cuda")
        elif kind == "normalize":
            s["x"] = _device_configurations(top, case["samples"], JITTER, seed)
            s["E"] = _labels(case["samples"], 1, seed)[0]
        elif kind == "train":
            n = case["batch"] * case["minibatches"]
            s["x"] = _device_configurations(top, n, JITTER, seed)
            s["E"], s["F"] = _labels(n, case["atoms"], seed)
            g = torch.Generator(device="cuda").manual_seed(seed + 3)
            s["perm"] = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
        else:
            r = case["replicas"]
            s["pop"] = pamd.Population(top, r, 600.0, seed, pamd.torch_options())
            s["pop"].set_state(_configurations(top, r, JITTER, seed), _velocities(top, r, 600.0, seed))
            surrogate.attach(s["pop"].ctx, s["model"])
    else:
        s["T"], E = _recorded(case, seed)
        s["E"] = torch.tensor(E, device="cuda")
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------ one pass

_REAL = ("T", "lnQ", "sum_lnQ", "e_pot", "e_pot_se", "e_kin", "e_kin_se", "t_meas", "rg", "rg_se", "rg2", "rg2_se")
_WHOLE = ("n_families", "max_copies", "R_live")


def _table(obs):
    """The observables of a run as one table of numbers and one of counts."""
    return {"averages": np.array([[o[k] for k in _REAL] for o in obs]),
            "counts": np.array([[o[k] for k in _WHOLE] for o in obs], np.int64)}


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "anneal":
        s["pop"].reset(case["t_first"], s["seed"])
        return _table(s["pop"].anneal(s["temps"], case["theta"], DT, resample=case["resample"]))
    if kind == "batch":
        pamd.pamd_reset(s["batch"].ctx, case["t_first"], s["seed"])
        obs = pamd.pamd_anneal(s["batch"].ctx, s["temps"], case["theta"], DT)
        return _table([o for at_T in obs for o in at_T])
    if kind == "fp64":
        s["pop"].propagate(case["theta"], DT, 600.0)
        x, v, E, _ = s["pop"].state()
        return {"x": x, "v": v, "E": E}
    if kind == "resample":
        # a program reads the counts and families of a population it inspects, not of a million replicas
        whole = case["replicas"] <= 65536
        copies, q0 = s["pop"].resample(1000.0, 985.0, want_copies=whole)
        _, q1 = s["pop"].resample(985.0, 1000.0, want_copies=False)
        out = {"lnQ": np.array([q0, q1]), **_table([s["pop"].observables(1000.0)])}
        if whole:
            _, _, E, fam = pamd.pamd_get_state(s["pop"].ctx, positions=False, velocities=False)
            out.update(copies=copies, E=E, fam=fam)
        return out
    if kind == "label":
        s["pop"].set_state(s["x"], s["v"])
        f, E = s["pop"].forces()
        return {"F": f.astype(np.float32), "E": E}
    if kind == "energy":
        if not case["autograd"]:
            E, F = s["model"].energy_forces(s["x"])
            return {"E": E, "F": F}
        x = s["x"].detach().requires_grad_(True)
        E = surrogate.surrogate_energy(x, s["model"])
        (gx,) = torch.autograd.grad(E, x, s["gE"])
        return {"E": E.detach(), "gx": gx}
    if kind == "train":
        model, b, losses = s["model"], case["batch"], None
        for k in range(case["minibatches"]):
            last = k == case["minibatches"] - 1
            losses = model.loss_grads(s["x"], s["E"], s["F"], idx=s["perm"][k * b:(k + 1) * b], sync=last)
            model.adam_step(1e-5)
        g = model.get_grads()
        return {"loss": losses, "W1": g["W1"], "b1": g["b1"], "W2": g["W2"], "b2": g["b2"], "w3": g["w3"],
                "b3": g["b3"]}
    if kind == "normalize":
        s["model"].fit_normalization(s["x"], s["E"])
        p = s["model"].get_params()
        return {k: p[k] for k in ("mu", "sd", "mu_E", "sigma_E")}
    if kind == "drive":
        s["pop"].propagate(case["theta"], DT, 600.0)
        o = s["pop"].observables(600.0)
        x, _, _, _ = pamd.pamd_get_state(s["pop"].ctx, velocities=False, energies=False, families=False)
        return {"x": x.astype(np.float32), "e_pot": o["e_pot"], "e_kin": o["e_kin"], "rg": o["rg"]}
    T = s["T"]
    return pamd.pamd_wham(s["E"].data_ptr(), len(T), case["replicas"], T, case["bins"], max_iter=case["sweeps"],
                          tol=1e-7, T_eval=np.sqrt(T[:-1] * T[1:]))


# ------------------------------------------------------------------ work

def _md_flops(n):
    """Flops of one BAOAB step of one replica: 40 a nonbonded pair, the bonded terms and the update."""
    pairs = max(n * (n - 1) // 2 - (2 * n - 3), 0)
    return 40 * pairs + 30 * (n - 1) + 60 * max(n - 2, 0) + 120 * max(n - 3, 0) + 20 * n


def work(case):
    kind = case["kind"]
    if kind == "anneal":
        n, r = case["atoms"], case["replicas"]
        return {"bytes": 48.0 * n * r, "flops": float(_md_flops(n)) * r * case["theta"] * (case["steps"] + 1)}
    if kind == "batch":
        sizes = pi.batched_chain_sizes(case["molecules"])
        r = case["replicas"]
        return {"bytes": 48.0 * sum(sizes) * r,
                "flops": float(sum(_md_flops(n) for n in sizes)) * r * case["theta"] * (case["steps"] + 1)}
    if kind == "fp64":
        n, r = case["atoms"], case["replicas"]
        return {"bytes": 96.0 * n * r, "flops": float(_md_flops(n)) * r * case["theta"]}
    if kind == "resample":
        n, r = case["atoms"], case["replicas"]
        # two gathers: state read and written, energies and families, copy counts
        return {"bytes": 2.0 * (48.0 * n + 24.0 + 4.0) * r, "flops": 0.0}
    if kind == "label":
        n, r = case["atoms"], case["replicas"]
        return {"bytes": (24.0 + 24.0 + 24.0) * n * r, "flops": float(_md_flops(n)) * r}
    if kind == "wham":
        nt, nb = case["temps"], case["bins"]
        # every sweep: an exponential of each bin and temperature, twice (about 25 flops each)
        return {"bytes": 8.0 * nt * case["replicas"], "flops": 50.0 * nt * nb * case["sweeps"]}
    n, h = case["atoms"], case["hidden"]
    p = n * (n - 1) // 2
    layer = 2.0 * h * (p + h)  # one pass through both layers for one sample
    if kind == "energy":
        m = case["samples"]
        return {"bytes": (24.0 * n + 8.0) * m + 2.0 * h * (p + h), "flops": 2 * layer * m}
    if kind == "train":
        m = case["batch"] * case["minibatches"]
        # forward, backward, tangent, its reverse, weight gradients over two operand sets
        return {"bytes": (24.0 * n + 8.0) * m + 28.0 * h * (p + h) * case["minibatches"], "flops": 6 * layer * m}
    if kind == "normalize":
        m = case["samples"]
        return {"bytes": (12.0 * n + 8.0) * m, "flops": 14.0 * p * m}
    return {"bytes": 48.0 * n * case["replicas"], "flops": 2 * layer * case["replicas"] * case["theta"]}


# ------------------------------------------------------------------ 64 bits

def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.asarray(a), device="cuda").to(dtype)


class _Field64:
    """The exact force field in 64 bits (autograd forces)."""

    def __init__(self, top):
        n = top.n_atoms
        self.n = n
        i, j = np.triu_indices(n, 1)
        lj, co = np.ones((n, n)), np.ones((n, n))
        for a, b in top.pair14:
            lj[a, b] = lj[b, a] = top.scale14_lj
            co[a, b] = co[b, a] = top.scale14_coul
        for a, b in top.excl:
            lj[a, b] = lj[b, a] = co[a, b] = co[b, a] = 0.0
        keep = (lj[i, j] != 0) | (co[i, j] != 0)
        i, j = i[keep], j[keep]
        self.i, self.j = _dev(i, torch.int64), _dev(j, torch.int64)
        self.sig2 = _dev((0.5 * (top.sigma[i] + top.sigma[j])) ** 2)
        self.eps4 = _dev(4.0 * np.sqrt(top.epsilon[i] * top.epsilon[j]) * lj[i, j])
        self.qq = _dev(KE * top.charge[i] * top.charge[j] * co[i, j])
        self.bond, self.angle, self.dih = (_dev(t, torch.int64) for t in (top.bond, top.angle, top.dihedral))
        self.b0, self.bk = _dev(top.bond_r0), _dev(top.bond_k)
        self.a0, self.ak = _dev(top.angle_t0), _dev(top.angle_k)
        self.dn, self.dk, self.dp = _dev(top.dih_n), _dev(top.dih_k), _dev(top.dih_phase)

    def energy(self, x):
        d = x[:, self.i] - x[:, self.j]
        r2 = (d * d).sum(-1)
        s6 = (self.sig2 / r2) ** 3
        e = (self.eps4 * (s6 * s6 - s6) + self.qq / r2.sqrt()).sum(-1)
        r = torch.linalg.vector_norm(x[:, self.bond[:, 0]] - x[:, self.bond[:, 1]], dim=-1)
        e = e + (0.5 * self.bk * (r - self.b0) ** 2).sum(-1)
        u = x[:, self.angle[:, 0]] - x[:, self.angle[:, 1]]
        w = x[:, self.angle[:, 2]] - x[:, self.angle[:, 1]]
        th = torch.atan2(torch.linalg.vector_norm(torch.cross(u, w, dim=-1), dim=-1), (u * w).sum(-1))
        e = e + (0.5 * self.ak * (th - self.a0) ** 2).sum(-1)
        b1 = x[:, self.dih[:, 1]] - x[:, self.dih[:, 0]]
        b2 = x[:, self.dih[:, 2]] - x[:, self.dih[:, 1]]
        b3 = x[:, self.dih[:, 3]] - x[:, self.dih[:, 2]]
        n1, n2 = torch.cross(b1, b2, dim=-1), torch.cross(b2, b3, dim=-1)
        phi = torch.atan2(torch.linalg.vector_norm(b2, dim=-1) * (b1 * n2).sum(-1), (n1 * n2).sum(-1))
        return e + (self.dk * (1.0 + torch.cos(self.dn * phi - self.dp))).sum(-1)

    def __call__(self, x):
        es, fs = [], []
        for c in x.split(max(1, (1 << 24) // (self.n * self.n))):
            c = c.detach().requires_grad_(True)
            with torch.enable_grad():
                e = self.energy(c)
                (g,) = torch.autograd.grad(e.sum(), c)
            es.append(e.detach())
            fs.append(-g)
        return torch.cat(es), torch.cat(fs)


class _Network64:
    """The surrogate in 64 bits with unrounded weights."""

    def __init__(self, w):
        self.t = {k: _dev(v) for k, v in w.items()}

    def e(self, x, t):
        a = (_features64(x) - self.t["mu"]) / self.t["sd"]
        silu = torch.nn.functional.silu
        return silu(silu(a @ t["W1"].T + t["b1"]) @ t["W2"].T + t["b2"]) @ t["w3"] + t["b3"]

    def __call__(self, x):
        es, fs = [], []
        for c in x.split(8192):
            c = c.detach().requires_grad_(True)
            e = self.e(c, self.t) * self.t["sigma_E"] + self.t["mu_E"]
            (g,) = torch.autograd.grad(e.sum(), c)
            es.append(e.detach())
            fs.append(-g)
        return torch.cat(es), torch.cat(fs)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _noise64(replicas, atoms, step, seed):
    slot = torch.arange(replicas, device="cuda")[:, None].expand(replicas, atoms)
    atom = torch.arange(atoms, device="cuda")[None, :].expand(replicas, atoms)
    o = _philox(atom, slot, torch.full_like(atom, step), torch.zeros_like(atom), seed)
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in o]
    r0, r1 = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    return torch.stack([r0 * torch.cos(2 * math.pi * u[1]), r0 * torch.sin(2 * math.pi * u[1]),
                        r1 * torch.cos(2 * math.pi * u[3])], -1)


def _baoab64(field, top, x, v, theta, T, seed):
    im = 1.0 / _dev(top.mass)[None, :, None]
    c1 = math.exp(-DT)
    sd = torch.sqrt((1.0 - c1 * c1) * KB * T * im)
    _, f = field(x)
    for k in range(theta):
        v = v + 0.5 * DT * f * im
        x = x + 0.5 * DT * v
        v = c1 * v + sd * _noise64(x.shape[0], x.shape[1], k, seed)
        x = x + 0.5 * DT * v
        e, f = field(x)
        v = v + 0.5 * DT * f * im
    return x, v, e


def exact(case, seed):
    kind = case["kind"]
    if kind in ("anneal", "batch", "resample"):
        return None  # averages over chaotic trajectories; copies and families are whole numbers
    if kind in ("fp64", "label"):
        top = _topology(case)
        x = _dev(_configurations(top, case["replicas"], JITTER_COLD, seed))
        if kind == "label":
            e, f = _Field64(top)(x)
            return {"F": f, "E": e}
        v = _dev(_velocities(top, case["replicas"], 600.0, seed))
        x, v, e = _baoab64(_Field64(top), top, x, v, case["theta"], 600.0, seed)
        return {"x": x, "v": v, "E": e}
    if kind == "wham":
        return _wham64(case, seed)
    top = pi.make_chain(case["atoms"], 1)
    if kind == "normalize":
        x = _device_configurations(top, case["samples"], JITTER, seed).double()
        g = torch.cat([_features64(c) for c in x.split(16384)])
        E = _labels(case["samples"], 1, seed)[0]
        return {"mu": g.mean(0), "sd": g.std(0, correction=0), "mu_E": float(E.mean()),
                "sigma_E": float(E.std(correction=0))}
    net = _Network64(_network(case, seed))
    if kind == "energy":
        E, F = net(_device_configurations(top, case["samples"], JITTER, seed).double())
        return {"E": E, "gx": -F} if case["autograd"] else {"E": E, "F": F}
    if kind == "drive":
        r = case["replicas"]
        x, v = _dev(_configurations(top, r, JITTER, seed)), _dev(_velocities(top, r, 600.0, seed))
        x, v, e = _baoab64(net, top, x, v, case["theta"], 600.0, seed)
        ek = (0.5 * _dev(top.mass)[None, :, None] * v * v).sum((1, 2))
        rg = (x - x.mean(1, keepdim=True)).square().sum(-1).mean(1).sqrt()
        return {"x": x, "e_pot": float(e.mean()), "e_kin": float(ek.mean()), "rg": float(rg.mean())}
    # train: the loss and its gradient, with Adam between the minibatches
    n, b, names = case["batch"] * case["minibatches"], case["batch"], ("W1", "b1", "W2", "b2", "w3", "b3")
    x = _device_configurations(top, n, JITTER, seed).double()
    E, F = _labels(n, case["atoms"], seed)
    perm = torch.randperm(n, generator=torch.Generator(device="cuda").manual_seed(seed + 3), device="cuda")
    t = {k: net.t[k].clone().requires_grad_(True) for k in names}
    m, q = ({k: torch.zeros_like(t[k]) for k in names} for _ in range(2))
    sE, muE = net.t["sigma_E"], net.t["mu_E"]
    for k in range(case["minibatches"]):
        idx = perm[k * b:(k + 1) * b]
        xs = x[idx].requires_grad_(True)
        e = net.e(xs, t)
        (g,) = torch.autograd.grad(e.sum(), xs, create_graph=True)
        df = -g - F[idx].double() / sE
        loss = ((e - (E[idx] - muE) / sE).square() + df.square().sum((1, 2)) / (3 * case["atoms"])).mean()
        grads = dict(zip(names, torch.autograd.grad(loss, [t[a] for a in names])))
        for a in names:
            m[a] = 0.9 * m[a] + 0.1 * grads[a]
            q[a] = 0.999 * q[a] + 0.001 * grads[a] ** 2
            step = (m[a] / (1 - 0.9 ** (k + 1))) / (torch.sqrt(q[a] / (1 - 0.999 ** (k + 1))) + 1e-8)
            t[a] = (t[a].detach() - 1e-5 * step).requires_grad_(True)
    out = {a: grads[a].detach() for a in names}
    return {"loss": float(loss.detach()), **out, "b3": float(out["b3"])}


def _logsumexp(a, axis):
    m = a.max(axis, keepdims=True)
    return np.squeeze(m + np.log(np.exp(a - m).sum(axis, keepdims=True)), axis)


def _wham64(case, seed):
    T, E = _recorded(case, seed)
    nb = case["bins"]
    beta, lo, hi = 1.0 / (KB * T), E.min(), E.max()
    width = (hi - lo) / nb
    at = np.clip(np.floor((E - lo) * (nb / (hi - lo))).astype(np.int64), 0, nb - 1)
    H = np.stack([np.bincount(a, minlength=nb) for a in at])
    N, total = H.sum(1), H.sum(0)
    Eb = lo + (np.arange(nb) + 0.5) * width
    used = total > 0
    lng, lnZ = np.full(nb, -np.inf), np.zeros(len(T))
    bE = beta[:, None] * Eb[None, used]

    def states():
        lng[used] = np.log(total[used]) - _logsumexp(np.log(N)[:, None] - bE - lnZ[:, None], 0)

    done, delta = 0, math.inf
    for _ in range(case["sweeps"]):
        states()
        new = _logsumexp(lng[None, used] - bE, 1)
        new -= new[0]
        delta, lnZ, done = float(np.abs(new - lnZ).max()), new, done + 1
        if delta < 1e-7:
            break
    states()
    Te = np.sqrt(T[:-1] * T[1:])
    a = lng[None, used] - Eb[None, used] / (KB * Te[:, None])
    z = _logsumexp(a, 1)
    p = np.exp(a - z[:, None])
    mean = (p * Eb[None, used]).sum(1)
    var = (p * (Eb[None, used] - mean[:, None]) ** 2).sum(1)
    return {"lnZ": lnZ, "ln_g": lng, "e_min": float(lo), "bin_width": float(width), "iterations": None,
            "max_delta": delta, "lnZ_eval": z, "e_mean_eval": mean, "e_var_eval": var}
