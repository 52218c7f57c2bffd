"""The calls a program makes of this framework, over the sizes it makes them at.

Every kind below goes through the package's public entry points the way a
program that uses them does: a batch of trials restored from a checkpoint and
advanced, the potential as a differentiable function of device tensors, the
reaction coordinate on its own, the functional's gradient along a path (given
frames, or a whole simulated path), descent on the functional, the similarity
of paths by the order their contacts form in, and the two-dimensional model.

`listed()` gives fixed cases, `draw(rng)` more of the same ranges, `prepare`
what the program holds before the call, `run` one call, `work` what the call
cannot do without and `exact` the same results from plain torch and numpy in
64 bits.
"""
import functools
import math

import numpy as np
import torch

from paper_1405_6104_gb300 import adjoint as A
from paper_1405_6104_gb300 import autograd as U
from paper_1405_6104_gb300 import binding as B
from paper_1405_6104_gb300 import systems as S

KB = 0.0083144626
FCOUL = 138.935458
EXACT_PAIRS = 5e10   # FP64 pair evaluations that take plain torch about 20 s
REFINE_STEP = 1e-8     # first step tried by a descent on the functional

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # a 1320-atom test system, one short call: launches and latency
        dict(name="steps_small", kind="steps", n_solute=60, n_water=420, n_systems=1, trials=1, steps=10, tuned=False),
        # one trial of the 11 040-atom system, launch shapes as they are by default
        dict(name="steps_single", kind="steps", n_solute=540, n_water=3500, n_systems=1, trials=1, steps=50, tuned=False),
        # the batch the benchmark times: 64 trials restored, advanced, scored, the best one read back
        dict(name="steps_batch", kind="steps", n_solute=540, n_water=3500, n_systems=1, trials=64, steps=20, tuned=True),
        # systems of uneven sizes in one batch (solutes and boxes differ by up to a factor of about ten)
        dict(name="steps_uneven", kind="steps", n_solute=247, n_water=2000, n_systems=7, trials=2, steps=20, tuned=True),
        # energy and forces of one configuration after another close by (a minimiser's or sampler's loop), FP64 tensors
        dict(name="potential_single", kind="potential", n_solute=540, n_water=3500, n_conf=1, dtype="float64", far=False),
        # new configurations scored in batches, FP32 tensors: every call needs new lists
        dict(name="potential_batch", kind="potential", n_solute=540, n_water=3500, n_conf=16, dtype="float32", far=True),
        # z and its gradient for one configuration, without device allocation: the smallest call
        dict(name="coordinate", kind="coordinate", n_cv=540),
        # gradient of the functional along one checkpoint segment of the 30 000-atom system's path
        dict(name="frames_gradient", kind="frames", n_cv=1800, n_frames=51),
        # descent on the functional from a short path of the 11 040-atom system's solute
        dict(name="refine", kind="refine", n_cv=540, n_frames=41, n_iter=6),
        # the functional's gradient along a simulated path of the 30 000-atom system, checkpointed replay
        dict(name="path_gradient", kind="path", n_solute=1800, n_water=9400, steps=500, every=50),
        # every pair of 64 trial paths, 23 160 native contacts
        dict(name="similarity", kind="similarity", n_paths=64, n_contacts=23160, n_times=11),
        # the two-dimensional model's rMD protocol: 2000 trials of 30 000 steps for each of four bias strengths
        dict(name="toy_rmd", kind="toy", n_trials=8000, n_steps=30000, bias=S.TOY_RATCHET, path_every=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "potential", "potential", "coordinate", "frames", "refine", "path",
                       "similarity", "toy"])
    if kind == "steps":
        n_sol, n_wat = _log_int(rng, 24, 1500), _log_int(rng, 480, 12000)
        n_sol = min(n_sol, n_wat // 4)
        n_systems = rng.choice([1, 1, 1, 2, 5])
        atoms = (n_sol + 3 * n_wat) * n_systems * (2 if n_systems > 1 else 1)
        trials = max(1, min(_log_int(rng, 1, 96), 700000 // atoms))
        steps = min(_log_int(rng, 5, 60), max(5, 14000000 // (atoms * trials)))
        return dict(kind=kind, n_solute=n_sol, n_water=n_wat, n_systems=n_systems, trials=trials, steps=steps,
                    tuned=rng.random() < 0.5)
    if kind == "potential":
        n_sol, n_wat = _log_int(rng, 24, 1500), _log_int(rng, 480, 9000)
        n_sol = min(n_sol, n_wat // 4)
        return dict(kind=kind, n_solute=n_sol, n_water=n_wat,
                    n_conf=max(1, min(_log_int(rng, 1, 24), 170000 // (n_sol + 3 * n_wat))),
                    dtype=rng.choice(["float32", "float64"]), far=rng.random() < 0.5)
    if kind == "coordinate":
        return dict(kind=kind, n_cv=_log_int(rng, 40, 2048))
    if kind == "frames":
        return dict(kind=kind, n_cv=_log_int(rng, 40, 1800), n_frames=_log_int(rng, 3, 60))
    if kind == "refine":
        return dict(kind=kind, n_cv=_log_int(rng, 40, 600), n_frames=_log_int(rng, 8, 48), n_iter=rng.randint(2, 6))
    if kind == "path":
        n_sol, n_wat = _log_int(rng, 24, 1500), _log_int(rng, 480, 8000)
        every = rng.choice([10, 25, 50])
        return dict(kind=kind, n_solute=min(n_sol, n_wat // 4), n_water=n_wat, steps=every * rng.randint(2, 8),
                    every=every)
    if kind == "similarity":
        # formation times are check steps: a few to some hundred distinct ones
        n_times = _log_int(rng, 4, 400)
        n_paths = _log_int(rng, 3, 64)
        n_c = _log_int(rng, 50, 24000 if n_times < 60 else 2500)
        return dict(kind=kind, n_paths=n_paths, n_contacts=n_c, n_times=n_times)
    n_steps = _log_int(rng, 200, 30000)
    bias = rng.choice([S.TOY_RATCHET, S.TOY_RATCHET, S.TOY_STEERED, S.TOY_NONE])
    return dict(kind="toy", n_trials=_log_int(rng, 30, 8000), n_steps=n_steps, bias=bias,
                path_every=0 if rng.random() < 0.7 else max(1, n_steps // 100))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


@functools.lru_cache(maxsize=64)
def _system(n_solute, n_water):
    """A solvated chain of this size (the geometry goes by the size alone)."""
    return S.solvated_heteropolymer(n_solute, n_water, seed=n_solute * 7919 + n_water)


def _systems(c):
    """The systems of a batch: one of the given size, or several whose solute
    and solvent grow by constant factors up to ten times the given size."""
    n = c.get("n_systems", 1)
    out = []
    for k in range(n):
        f = 10.0 ** (k / n)
        n_wat = int(round(c["n_water"] * f))
        out.append(_system(min(int(round(c["n_solute"] * f ** 0.8)), n_wat // 4), n_wat))
    return out


def _params(n_solute, k_ratchet=None):
    """Parameters of the solvated chains; short chains count contacts from a
    smaller separation and take a stiffer ratchet, as the test systems do."""
    p = S.protein_params(1)
    if n_solute < 200:
        p.k_ratchet, p.cv_min_sep = 5.0, 4
    if k_ratchet is not None:
        p.k_ratchet = k_ratchet
    return p


def _f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def _velocities(s, rng, temperature=300.0):
    sd = np.sqrt(KB * temperature / np.asarray(s.mass))[:, None]
    v = sd * rng.normal(size=(s.n_atoms, 3))
    v -= (s.mass[:, None] * v).sum(0) / s.mass.sum()
    return _f32(v)


def _path_frames(n_cv, n_frames, rng):
    """(system, FP32-valued frames of a partly folded chain): it moves towards
    the fold and back by some hundredths of a nanometre, with thermal noise,
    so z falls and rises and the ratchet acts."""
    s = _system(n_cv, max(480, 3 * n_cv))
    nat, x0 = s.native_pos, s.pos[:n_cv].copy()
    # the starting coil is stored wrapped into the box: make the chain whole
    for i in range(1, n_cv):
        x0[i] -= s.box * np.round((x0[i] - x0[i - 1]) / s.box)
    t = 0.8 + rng.uniform(-0.1, 0.1) + 0.002 * np.cos(np.linspace(0.0, 2.5 * math.pi, n_frames))
    fr = np.stack([nat + u * (x0 - nat) + 0.0005 * rng.normal(size=nat.shape) for u in t])
    return s, _f32(fr)


def _similarity_times(c, rng):
    """Formation times as the tracker gives them: multiples of the check
    interval, most contacts formed early, some never (-1); the paths share an
    order with their own deviations."""
    base = rng.gamma(1.5, 0.25, size=c["n_contacts"])
    t = base[None] * np.exp(0.35 * rng.normal(size=(c["n_paths"], c["n_contacts"])))
    k = np.minimum((t / 1.2 * c["n_times"]).astype(np.int64) + 1, c["n_times"])
    k[rng.random(k.shape) < 0.04] = -1
    return np.where(k < 0, -1, 10 * k)


def _path_pairs(n):
    return np.array([(a, b) for a in range(n) for b in range(a + 1, n)], np.int32).reshape(-1, 2)


def _toy(c, rng):
    n = c["n_trials"]
    ks = np.repeat([0.5, 1.0, 4.0, 16.0], (n + 3) // 4)[:n]
    return S.Toy2dParams(bias=c["bias"]), ks, rng.integers(1, 2 ** 40, size=n).astype(np.uint64)


def _coordinate(c, rng):
    """(system, parameters, FP32-valued frame): a partly folded chain."""
    s, fr = _path_frames(c["n_cv"], 3, rng)
    return s, _params(c["n_cv"]), fr[1]


def _steps_inputs(c, seed):
    rng = np.random.default_rng(seed)
    systems = _systems(c)
    tps = [c["trials"]] * len(systems)
    per = [s for s, n in zip(systems, tps) for _ in range(n)]
    pos = np.concatenate([_f32(s.pos) for s in per])
    vel = np.concatenate([_velocities(s, rng) for s in per])
    seeds = [int(x) for x in rng.integers(1, 2 ** 40, size=len(per))]
    return systems, tps, per, pos, vel, seeds, _params(c["n_solute"])


def _potential_inputs(c, seed):
    """Configurations around the generated one; with `far`, a second set far
    enough from the first that the lists of one do not serve the other."""
    rng = np.random.default_rng(seed)
    s = _system(c["n_solute"], c["n_water"])
    n_sets = 2 if c["far"] else 1
    conf = s.pos[None, None] + 0.003 * rng.normal(size=(n_sets, c["n_conf"], s.n_atoms, 3))
    conf[1:] += 0.08
    return s, _params(c["n_solute"]), _f32(conf)


def prepare(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    dev = torch.device("cuda")
    if c["kind"] == "steps":
        systems, tps, per, pos, vel, seeds, p = _steps_inputs(c, seed)
        batch = B.TrialBatch(systems, p, tps, trial_seeds=seeds)
        if c["tuned"]:
            B.sim_autotune(batch.h, 5, None)
            B.sim_autotune_step(batch.h, 2)
        return dict(c, batch=batch, pos=pos, vel=vel)
    if c["kind"] == "potential":
        s, p, conf = _potential_inputs(c, seed)
        t = torch.tensor(conf, dtype=getattr(torch, c["dtype"]), device=dev)
        w = torch.tensor(rng.normal(size=(len(conf), c["n_conf"])), dtype=t.dtype, device=dev)
        return dict(c, evaluator=U.Evaluator(s, p, n_conf=c["n_conf"]), sets=list(t), weights=list(w))
    if c["kind"] == "coordinate":
        s, p, x = _coordinate(c, rng)
        return dict(c, params=p, box=s.box, pos=torch.tensor(x, dtype=torch.float32, device=dev).reshape(-1).contiguous(),
                    native=torch.tensor(s.native_pos, dtype=torch.float64, device=dev).reshape(-1).contiguous())
    if c["kind"] == "frames":
        s, fr = _path_frames(c["n_cv"], c["n_frames"], rng)
        return dict(c, batch=B.TrialBatch(s, _params(c["n_cv"], 5.0), [1]), frames=fr)
    if c["kind"] == "refine":
        s, fr = _path_frames(c["n_cv"], c["n_frames"], rng)
        return dict(c, batch=B.TrialBatch(s, _params(c["n_cv"], 5.0), [1]), frames=fr)
    if c["kind"] == "path":
        s = _system(c["n_solute"], c["n_water"])
        pos, vel = _f32(s.pos), _velocities(s, rng)
        batch = B.TrialBatch(s, _params(c["n_solute"], 5.0), [1], trial_seeds=[int(rng.integers(1, 2 ** 40))])
        B.sim_autotune(batch.h, 3, None)
        B.sim_autotune_step(batch.h, 2)
        st = dict(c, batch=batch, pos=pos, vel=vel)
        run(st)  # the batch that replays the segments is made at the first call and kept with this one
        return st
    if c["kind"] == "similarity":
        return dict(c, times=_similarity_times(c, rng), pairs=_path_pairs(c["n_paths"]))
    tp, ks, seeds = _toy(c, rng)
    return dict(c, tp=tp, ks=ks, seeds=seeds)


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------


def _best(phi, n_systems):
    """The least functional of each system's trials (equal numbers of them)."""
    per = len(phi) // n_systems
    return np.arange(n_systems) * per + np.argmin(np.reshape(phi, (n_systems, per)), axis=1)


def run(state):
    st = state
    if st["kind"] == "steps":
        # restored from a checkpoint, advanced, scored, the optimum read back
        b = st["batch"]
        B.sim_set_step_count(b.h, 0)
        b.set_state(-1, st["pos"], st["vel"])
        b.step(st["steps"])
        phi, best = b.bias_functional()
        if st["n_systems"] > 1:  # one optimum per system
            best = _best(phi, st["n_systems"])
            return {"phi": phi, "best": best, "states": [b.get_state(int(t)) for t in best]}
        pos, vel, cv = b.get_state(best)
        return {"phi": phi, "best": best, "pos": pos, "vel": vel, "cv": cv}
    if st["kind"] == "potential":
        out = []
        for x, w in zip(st["sets"], st["weights"]):
            x = x.clone().requires_grad_(True)
            u = U.potential_energy(x, st["evaluator"])
            (u * w).sum().backward()
            out.append((u.detach(), x.grad))
        return out
    if st["kind"] == "coordinate":
        z = torch.empty(1, dtype=torch.float64, device="cuda")
        g = torch.empty(3 * st["n_cv"], dtype=torch.float64, device="cuda")
        rc, msg = B.cv_eval_noalloc(st["pos"].data_ptr(), st["native"].data_ptr(), st["n_cv"], st["box"], st["params"],
                                    z.data_ptr(), g.data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != B.SIM_OK:
            raise RuntimeError(msg)
        return {"z": z, "grad": g}
    if st["kind"] == "frames":
        phi, z, g = B.phi_frames_adjoint(st["batch"].h, 0, st["frames"])
        return {"phi": phi, "z": z, "grad": g}
    if st["kind"] == "refine":
        x, hist, acc = B.phi_frames_refine(st["batch"].h, 0, st["frames"], st["n_iter"], REFINE_STEP)
        return {"frames": x, "phi": hist, "accepted": acc}
    if st["kind"] == "path":
        b = st["batch"]
        B.sim_set_step_count(b.h, 0)
        b.set_state(-1, st["pos"], st["vel"])
        phi, grad, info = A.trajectory_adjoint(b, 0, st["steps"], every=st["every"])
        return {"phi": phi, "grad": grad, "z": info["z"]}
    if st["kind"] == "similarity":
        return B.path_similarity(st["times"], st["pairs"])
    passage, phi, end, path = B.toy2d_run(st["tp"], st["ks"], st["seeds"], st["n_steps"], path_every=st["path_every"])
    return {"passage": passage, "phi": phi, "state": end, "path": path}


# ---------------------------------------------------------------------------
# what a call cannot do without
# ---------------------------------------------------------------------------


def _cv_pairs(n, sep):
    m = max(0, n - sep - 1)
    return m * (m + 1) / 2


def _half_pairs(s, r):
    """Pairs inside r per atom of a homogeneous system."""
    return 0.5 * 4.0 / 3.0 * math.pi * r ** 3 * s.n_atoms / s.box ** 3


def _sep(n_solute):
    return _params(n_solute).cv_min_sep


def work(case):
    """Pair interactions 35 operations, contact pairs 10 by distance alone
    (most are farther than the cut-off), the two-dimensional model 109 a step."""
    c = case
    if c["kind"] in ("steps", "path"):
        systems, trials = _systems(c), c.get("trials", 1)
        # the checkpoint goes in (FP64 positions and velocities); Phi per trial and one trial's state come out
        steps = c["steps"] * (2 if c["kind"] == "path" else 1)  # the path is run again from its checkpoints
        flops = sum(s.n_atoms * (35.0 * _half_pairs(s, 1.0) + 100.0) + 10.0 * _cv_pairs(s.n_cv, _sep(c["n_solute"]))
                    for s in systems) * trials * steps
        bytes_ = sum(48.0 * s.n_atoms for s in systems) * trials + 48.0 * max(s.n_atoms for s in systems)
        if c["kind"] == "path":
            bytes_ += 24.0 * c["n_solute"] * (c["steps"] + 1)
            flops += 60.0 * _cv_pairs(c["n_solute"], _sep(c["n_solute"])) * c["steps"]
        return {"bytes": bytes_, "flops": flops}
    if c["kind"] == "potential":
        s = _system(c["n_solute"], c["n_water"])
        n = s.n_atoms * c["n_conf"] * (2 if c["far"] else 1)
        return {"bytes": n * 6.0 * (8 if c["dtype"] == "float64" else 4), "flops": n * 45.0 * _half_pairs(s, 1.0)}
    if c["kind"] == "coordinate":
        return {"bytes": c["n_cv"] * (12.0 + 24.0 + 24.0), "flops": 20.0 * _cv_pairs(c["n_cv"], _sep(c["n_cv"]))}
    if c["kind"] == "frames":
        return {"bytes": 48.0 * c["n_cv"] * c["n_frames"],
                "flops": 60.0 * _cv_pairs(c["n_cv"], _sep(c["n_cv"])) * c["n_frames"]}
    if c["kind"] == "refine":
        return {"bytes": 48.0 * c["n_cv"] * c["n_frames"],
                "flops": 80.0 * _cv_pairs(c["n_cv"], _sep(c["n_cv"])) * c["n_frames"] * (c["n_iter"] + 1)}
    if c["kind"] == "similarity":
        pairs = c["n_paths"] * (c["n_paths"] - 1) / 2
        return {"bytes": 8.0 * c["n_paths"] * c["n_contacts"] + 16.0 * pairs, "flops": 2.0 * pairs * c["n_contacts"]}
    n = c["n_trials"]
    return {"bytes": n * (16.0 + 48.0) + (16.0 * n * (c["n_steps"] // c["path_every"] + 1) if c["path_every"] else 0.0),
            "flops": 109.0 * n * c["n_steps"]}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------


def _t(a, dtype=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


class _Exact:
    """U, -grad U and the reaction coordinate of one system in FP64."""

    def __init__(self, s, p):
        self.s, self.p = s, p
        self.L = float(np.float32(s.box))
        n = s.n_atoms
        self.q, self.m = _t(s.charge) * math.sqrt(FCOUL), _t(s.mass)
        ty = torch.tensor(np.asarray(s.lj_type), dtype=torch.int64, device="cuda")
        sig, eps = _t(s.sigma), _t(s.epsilon)
        self.sig, self.eps = sig[ty], torch.sqrt(eps)[ty]
        ex = {(min(a, b), max(a, b)) for a, b in np.asarray(s.bonds).tolist()}
        ex |= {(min(a, c), max(a, c)) for a, _, c in np.asarray(s.angles).tolist()}
        e = torch.tensor(sorted(ex), dtype=torch.int64, device="cuda").reshape(-1, 2)
        self.exc = torch.cat([e, e.flip(1)])
        self.bonds = torch.tensor(np.asarray(s.bonds), dtype=torch.int64, device="cuda").reshape(-1, 2)
        self.angles = torch.tensor(np.asarray(s.angles), dtype=torch.int64, device="cuda").reshape(-1, 3)
        self.b0, self.bk, self.a0, self.ak = (_t(v) for v in (s.bond_r0, s.bond_k, s.angle_t0, s.angle_k))
        self.krf, self.crf = 1.0 / (2.0 * p.r_cut ** 3), 3.0 / (2.0 * p.r_cut)
        self.rows = max(1, min(n, int(3e7) // n))
        i, j = torch.triu_indices(s.n_cv, s.n_cv, p.cv_min_sep + 1, device="cuda")
        self.ci, self.cj = i, j
        nat = _t(s.native_pos)
        self.cnat = self._contact(((nat[j] - nat[i]) ** 2).sum(1))
        g = p.gamma if s.gamma is None else _t(s.gamma)
        self.inv_gm = (1.0 / (g * self.m))[: s.n_cv]

    def _image(self, d):
        return d - self.L * torch.round(d / self.L)

    def potential(self, x):
        """(U, F) at x (n, 3)."""
        n, p = len(x), self.p
        F = torch.zeros_like(x)
        E = torch.zeros((), dtype=torch.float64, device="cuda")
        cols = torch.arange(n, device="cuda")
        for a in range(0, n, self.rows):
            b = min(n, a + self.rows)
            d = self._image(x[None, :, :] - x[a:b, None, :])
            r2 = (d * d).sum(2)
            keep = (r2 < p.r_cut ** 2) & (cols[None] != cols[a:b, None])
            sel = (self.exc[:, 0] >= a) & (self.exc[:, 0] < b)
            keep[self.exc[sel, 0] - a, self.exc[sel, 1]] = False
            i, j = keep.nonzero(as_tuple=True)
            d, r2, i = d[i, j], r2[i, j], i + a
            sig, eps, qq = 0.5 * (self.sig[i] + self.sig[j]), self.eps[i] * self.eps[j], self.q[i] * self.q[j]
            s6 = (sig * sig / r2) ** 3
            c6 = (sig / p.r_cut) ** 6
            rinv = 1.0 / torch.sqrt(r2)
            E = E + 0.5 * (4.0 * eps * (s6 * s6 - s6 - c6 * c6 + c6) + qq * (rinv + self.krf * r2 - self.crf)).sum()
            f = (24.0 * eps * (2.0 * s6 * s6 - s6) + qq * rinv) / r2 - 2.0 * self.krf * qq
            F.index_add_(0, i, -f[:, None] * d)
        xb = x.detach().clone().requires_grad_(True)
        d = self._image(xb[self.bonds[:, 1]] - xb[self.bonds[:, 0]])
        eb = (0.5 * self.bk * (d.norm(dim=1) - self.b0) ** 2).sum()
        if len(self.angles):
            u = self._image(xb[self.angles[:, 0]] - xb[self.angles[:, 1]])
            v = self._image(xb[self.angles[:, 2]] - xb[self.angles[:, 1]])
            cs = (u * v).sum(1) / (u.norm(dim=1) * v.norm(dim=1))
            eb = eb + (0.5 * self.ak * (torch.acos(cs) - self.a0) ** 2).sum()
        (g,) = torch.autograd.grad(eb, xb)
        return E + eb.detach(), F - g

    def _contact(self, r2):
        p = self.p
        s = r2 / p.cv_r0 ** 2
        c = (1 + s + s * s) / (1 + s + s * s + s ** 3 + s ** 4)
        x = ((torch.sqrt(r2) - p.cv_r_switch) / (p.cv_r_cut - p.cv_r_switch)).clamp(0.0, 1.0)
        return c * (1.0 - x ** 3 * (10.0 - 15.0 * x + 6.0 * x * x))

    def z(self, x):
        d = self._image(x[self.cj] - x[self.ci])
        return ((self._contact((d * d).sum(1)) - self.cnat) ** 2).sum()

    def z_grad(self, x):
        y = x[: self.s.n_cv].detach().clone().requires_grad_(True)
        z = self.z(y)
        return z.detach(), torch.autograd.grad(z, y)[0]

    def z_Q(self, x):
        z, g = self.z_grad(x)
        return float(z), float(((g * g).sum(1) * self.inv_gm).sum())

    def coefficients(self, z, Q):
        """(Phi, A_n, c a_n^2) of dPhi/dX_n = A_n grad z + c a_n^2 grad Q."""
        c = self.p.dt * (0.5 * self.p.k_ratchet) ** 2
        n = len(z)
        route, A_, B_ = np.zeros(n), np.zeros(n), np.zeros(n)
        m, arg, phi = z[0], 0, 0.0
        for f in range(1, n):
            a = max(z[f] - m, 0.0)
            phi += c * a * a * Q[f]
            route[arg] += 2.0 * a * Q[f]
            A_[f], B_[f] = 2.0 * c * a * Q[f], c * a * a
            if z[f] < m:
                m, arg = z[f], f
        return phi, A_ - c * route, B_

    def phi(self, frames):
        zq = [self.z_Q(x) for x in frames]
        z, Q = np.array([v[0] for v in zq]), np.array([v[1] for v in zq])
        phi, A_, B_ = self.coefficients(z, Q)
        return phi, z, A_, B_

    def phi_grad(self, frames):
        phi, z, A_, B_ = self.phi(frames)
        out = []
        for x, a, b in zip(frames, A_, B_):
            y = x.detach().clone().requires_grad_(True)
            v = self.z(y)
            if b == 0.0:
                out.append(torch.autograd.grad(a * v, y)[0])
                continue
            (g,) = torch.autograd.grad(v, y, create_graph=True)
            q = ((g * g).sum(1) * self.inv_gm).sum()
            out.append(torch.autograd.grad(a * v + b * q, y)[0])
        return phi, z, torch.stack(out)


def _philox(n, step, stream, seed):
    """Philox4x32-10 of the counters (atom, step, stream): (4, n) words."""
    m32 = np.uint64(0xFFFFFFFF)
    c = [np.arange(n, dtype=np.uint64), np.full(n, step & 0xFFFFFFFF, np.uint64), np.full(n, step >> 32, np.uint64),
         np.full(n, stream, np.uint64)]
    k0, k1 = np.asarray(seed, np.uint64) & m32, np.asarray(seed, np.uint64) >> np.uint64(32)
    if np.ndim(seed):  # one counter 0 per seed
        c[0] = np.zeros(n, np.uint64)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m32]
    return np.stack(c)


def _uniforms(words):
    return ((words >> np.uint64(9)).astype(np.float64) + 0.5) / 8388608.0


def _noise(n, step, seed):
    u = _uniforms(_philox(n, step, 0, seed))
    r, q = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    return np.stack([r * np.cos(2 * np.pi * u[1]), r * np.sin(2 * np.pi * u[1]), q * np.cos(2 * np.pi * u[3])], 1)


def _trajectory(ex, pos, vel, seed, steps, forced=0, keep=None):
    """`steps` steps of one trial from (pos, vel): (x, v, [z, z_m, a, Phi]).
    Positions are wrapped into the box where its pair list is rebuilt: at the
    start, when an atom has moved half the buffer, after nstlist steps, and
    every `forced` steps.  keep(x) sees every frame."""
    s, p = ex.s, ex.p
    n, L, dt = s.n_atoms, ex.L, p.dt
    x, v = _t(pos), _t(vel)
    m = ex.m[:, None]
    c1 = math.exp(-p.gamma * dt)
    sd = torch.sqrt((1.0 - c1 * c1) * KB * p.temperature / m)
    trig = (0.5 * p.skin - 1e-5) ** 2
    wrap = lambda y: y - L * torch.floor(y / L)  # noqa: E731
    x = wrap(x)
    ref, last = x.clone(), 0
    z, g = ex.z_grad(x)
    zm, a, phi = float(z), 0.0, 0.0
    if keep:
        keep(x)
    F = ex.potential(x)[1]
    for k in range(1, steps + 1):
        v = v + 0.5 * dt * F / m
        x = x + 0.5 * dt * v
        v = c1 * v + sd * _t(_noise(n, k, seed))
        x = x + 0.5 * dt * v
        if float(((x - ref) ** 2).sum(1).max()) > trig or k - last >= p.nstlist:
            x = wrap(x)
            ref, last = x.clone(), k
        F = ex.potential(x)[1]
        z, g = ex.z_grad(x)
        a = max(float(z) - zm, 0.0)
        phi += dt * (0.5 * p.k_ratchet * a) ** 2 * float(((g * g).sum(1) * ex.inv_gm).sum())
        zm = min(zm, float(z))
        F[: s.n_cv] -= 0.5 * p.k_ratchet * a * g
        if keep:
            keep(x)
        v = v + 0.5 * dt * F / m
        if forced and k % forced == 0:
            x = wrap(x)
            ref, last = x.clone(), k
    return x, v, np.array([float(z), zm, a, phi])


def _exact_toy(tp, ks, seeds, n_steps, every):
    n = len(ks)
    p = 4 if tp.s_power == 4 else 2

    def normals(step, stream):
        u = _uniforms(_philox(n, step, stream, seeds))
        r = np.sqrt(-2.0 * np.log(u[0]))
        return r * np.cos(2 * np.pi * u[1]), r * np.sin(2 * np.pi * u[1])

    def force(x, y):
        r2 = x * x + y * y
        q = 4 * tp.w ** 2 * r2
        q = q + 4 * tp.A1 * tp.s1 ** p / (r2 + tp.s1 ** 2) ** 3 - 4 * tp.A2 * tp.s2 ** p / (r2 + tp.s2 ** 2) ** 3
        dx, dy = x - tp.xm, y - tp.ym
        g = 4 * tp.A3 * tp.s3 ** p / (dx * dx + dy * dy + tp.s3 ** 2) ** 3
        return -q * x - g * dx, -q * y - g * dy

    def bias(x, y, z, zm):
        zz = np.where(z == 0.0, 1.0, z)
        f = -0.5 * ks * np.maximum(z - zm, 0.0) if tp.bias == S.TOY_RATCHET else -ks * z if tp.bias == S.TOY_STEERED else 0.0 * z
        return f * x / zz, f * y / zz

    h, c1, sd = 0.5 * tp.dt, math.exp(-tp.gamma * tp.dt), math.sqrt(tp.kT / tp.mass)
    c2 = math.sqrt(1.0 - c1 * c1) * sd
    x, y = np.full(n, tp.x0), np.full(n, tp.y0)
    g = normals(0, 1)
    vx, vy = sd * g[0], sd * g[1]
    zm = np.hypot(x, y)
    F = [a + b for a, b in zip(force(x, y), bias(x, y, zm, zm))]
    phi, passage = np.zeros(n), np.full(n, -1, np.int64)
    path = np.full((n, n_steps // every + 1, 2), np.nan) if every else None
    if every:
        path[:, 0, 0], path[:, 0, 1] = x, y
    for s in range(1, n_steps + 1):
        on = passage < 0
        if not on.any():
            break
        g = normals(s, 0)
        nvx, nvy = vx + h * F[0] / tp.mass, vy + h * F[1] / tp.mass
        nx, ny = x + h * nvx, y + h * nvy
        nvx, nvy = c1 * nvx + c2 * g[0], c1 * nvy + c2 * g[1]
        nx, ny = nx + h * nvx, ny + h * nvy
        z = np.hypot(nx, ny)
        b = bias(nx, ny, z, zm)
        nF = [p_ + q_ for p_, q_ in zip(force(nx, ny), b)]
        nvx, nvy = nvx + h * nF[0] / tp.mass, nvy + h * nF[1] / tp.mass
        phi = np.where(on, phi + tp.dt * (b[0] ** 2 + b[1] ** 2) / (tp.gamma * tp.mass), phi)
        x, y, vx, vy = (np.where(on, a, o) for a, o in ((nx, x), (ny, y), (nvx, vx), (nvy, vy)))
        F = [np.where(on, a, o) for a, o in zip(nF, F)]
        zm = np.where(on, np.minimum(zm, z), zm)
        if every and s % every == 0:
            path[on, s // every, 0], path[on, s // every, 1] = x[on], y[on]
        passage[on & (z <= tp.z_product)] = s
    return {"passage": passage, "phi": phi, "state": np.stack([x, y, vx, vy], 1), "path": path}


def exact(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    if c["kind"] == "steps":
        systems, tps, per, pos, vel, seeds, p = _steps_inputs(c, seed)
        if sum(float(s.n_atoms) ** 2 for s in per) * (c["steps"] + 1) > EXACT_PAIRS:
            return None
        got, at, made = [], 0, {}
        for s, sd in zip(per, seeds):
            ex = made.setdefault(id(s), None) or _Exact(s, p)
            made[id(s)] = ex
            got.append(_trajectory(ex, pos[at:at + s.n_atoms], vel[at:at + s.n_atoms], sd, c["steps"]))
            at += s.n_atoms
        phi = np.array([g[2][3] for g in got])
        if c["n_systems"] > 1:
            best = _best(phi, c["n_systems"])
            return {"phi": phi, "best": best, "states": [got[t] for t in best]}
        best = int(np.argmin(phi))
        return {"phi": phi, "best": best, "pos": got[best][0], "vel": got[best][1], "cv": got[best][2]}
    if c["kind"] == "potential":
        s, p, conf = _potential_inputs(c, seed)
        if float(s.n_atoms) ** 2 * conf.shape[0] * conf.shape[1] > EXACT_PAIRS:
            return None
        w = rng.normal(size=(len(conf), c["n_conf"]))
        w = _t(w, getattr(torch, c["dtype"])).double()
        ex, out = _Exact(s, p), []
        for k in range(len(conf)):
            ef = [ex.potential(_t(x)) for x in conf[k]]
            out.append((torch.stack([e for e, _ in ef]), torch.stack([-w[k, i] * f for i, (_, f) in enumerate(ef)])))
        return out
    if c["kind"] == "coordinate":
        s, p, x = _coordinate(c, rng)
        z, g = _Exact(s, p).z_grad(_t(x))
        return {"z": z.reshape(1), "grad": g.reshape(-1)}
    if c["kind"] == "frames":
        s, fr = _path_frames(c["n_cv"], c["n_frames"], rng)
        phi, z, g = _Exact(s, _params(c["n_cv"], 5.0)).phi_grad(_t(fr))
        return {"phi": phi, "z": z, "grad": g}
    if c["kind"] == "refine":
        s, fr = _path_frames(c["n_cv"], c["n_frames"], rng)
        ex = _Exact(s, _params(c["n_cv"], 5.0))
        x, eta, acc = _t(fr), REFINE_STEP, 0
        phi, _, g = ex.phi_grad(x)
        hist = [phi]
        for _ in range(c["n_iter"]):
            g[0] = g[-1] = 0.0
            gg, ok = float((g * g).sum()), False
            for _ in range(40 if gg > 0.0 else 0):
                y = x.clone()
                y[1:-1] = (x - eta * g)[1:-1].float().double()
                phi_y = ex.phi(y)[0]
                if phi_y <= phi - 1e-4 * eta * gg:
                    x, phi, ok = y, phi_y, True
                    break
                eta *= 0.5
            if not ok:
                break
            phi, _, g = ex.phi_grad(x)
            acc, eta = acc + 1, 2.0 * eta
            hist.append(phi)
        return {"frames": x, "phi": np.array(hist + [hist[-1]] * (c["n_iter"] + 1 - len(hist))), "accepted": acc}
    if c["kind"] == "path":
        s = _system(c["n_solute"], c["n_water"])
        if float(s.n_atoms) ** 2 * c["steps"] > EXACT_PAIRS:
            return None
        pos, vel = _f32(s.pos), _velocities(s, rng)
        ex, frames = _Exact(s, _params(c["n_solute"], 5.0)), []
        _trajectory(ex, pos, vel, int(rng.integers(1, 2 ** 40)), c["steps"], forced=c["every"],
                    keep=lambda x: frames.append(x[: s.n_cv].clone()))
        phi, z, g = ex.phi_grad(torch.stack(frames))
        return {"phi": phi, "grad": g, "z": z}
    if c["kind"] == "similarity":
        t = _similarity_times(c, rng)
        t = np.where(t < 0, np.iinfo(np.int64).max, t)
        rank = [np.unique(row, return_inverse=True)[1] for row in t]
        n, out = c["n_contacts"], []
        for a, b in _path_pairs(c["n_paths"]):
            ka, kb = rank[a].max() + 1, rank[b].max() + 1
            h = np.bincount(rank[a] * kb + rank[b], minlength=ka * kb).reshape(ka, kb).astype(np.float64)
            below = np.zeros_like(h)
            below[1:, 1:] = h.cumsum(0).cumsum(1)[:-1, :-1]
            out.append(((h * (h - 1)).sum() + 2.0 * (h * below).sum()) / (n * (n - 1.0)))
        return np.array(out)
    if c["n_steps"] > 3000:  # rounding grows to the size of the path: the end has no value of its own
        return None
    tp, ks, seeds = _toy(c, rng)
    return _exact_toy(tp, ks, seeds, c["n_steps"], c["path_every"])
