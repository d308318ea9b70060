"""Timed workloads of the time stepper, called as a user's program calls it.

Sizes and parameters are those of workloads.CONFIGS (c1, c2, c3, c5, n1e5, the
batched replicas) and of the tests' ragged sizes.  Each case names one kind of
call:

  steps      advance `steps` time steps, then read the state into page-locked
             host arrays (a simulation that keeps every so many snapshots)
  coupled    set the state, one step, read the state (another program on the
             host owns the state between steps)
  batch      the same as steps for an ensemble of independent replicas
  gradient   a recorded rollout and its reverse pass through the autograd
             wrapper, with single-precision parameters as an optimiser keeps
  forces     the pair force at the current positions (analysis of a state)
  noalloc    the pair force on tensors that the caller's allocator owns

The FP32 path's forces and gradients are returned in single precision: that is
the precision the step itself reads them in, and what a program goes on with.
Positions, directions and the FP64 path's results are returned as they come.
"""
import math

import numpy as np
import torch

import paper_1703_02484_gb300 as bd
from paper_1703_02484_gb300 import binding, workloads

CONFIG = workloads.CONFIGS

# the largest work of a drawn case: ordered pairs per pass of the all-pairs
# laws, disk-steps of the short-range ones
MOST_PAIRS = 2.0e10
MOST_DISK_STEPS = 1.6e7


def listed():
    return [
        # the smallest call: a small active system driven from the host step by
        # step, where launches, synchronisations and copies count
        dict(name="coupled_777", kind="coupled", config="c2", n=777, periodic=False),
        # the FP64 path at the size of the passive one-species configuration
        dict(name="c1_fp64_1024", kind="steps", config="c1", n=1024, steps=20, periodic=False),
        # the two-species active configuration, walls, FP32
        dict(name="c2_16384", kind="steps", config="c2", n=16384, steps=20, periodic=False),
        # the throughput workload: 1e5 disks, every pair, walls
        dict(name="n1e5", kind="steps", config="n1e5", n=100000, steps=2, periodic=False),
        # the paper's periodic box with the long-range law, a ragged size
        dict(name="periodic_30011", kind="steps", config="n1e5", n=30011, steps=5, periodic=True),
        # the short-range law at the largest size, overlaps over the Delaunay edges
        dict(name="c3_1048576", kind="steps", config="c3", n=1048576, steps=10, periodic=False),
        # the short-range law with overlaps over the Verlet lists, periodic box
        dict(name="verlet_200003", kind="steps", config="c3", n=200003, steps=20, periodic=True, verlet=True),
        # slightly polydisperse disks, short-range law
        dict(name="poly_20000", kind="steps", config="c3", n=20000, steps=20, periodic=False, ratio=1.3),
        # an ensemble of independent systems of mixed sizes, densities and laws
        dict(name="batch_64", kind="batch", replicas=64, n_lo=512, n_hi=16384, steps=4),
        # gradients of a rollout's loss, forward and reverse
        dict(name="gradient_4096", kind="gradient", config="c5", n=4096, steps=40, ckpt=20, loss="msd"),
        # forces of a state for analysis, a size between the configurations'
        dict(name="forces_20011", kind="forces", config="c2", n=20011, periodic=False),
        # forces on a host framework's own tensors, a ragged size
        dict(name="noalloc_30011", kind="noalloc", n=30011),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["coupled", "steps", "steps", "steps", "short", "short", "batch", "gradient", "forces", "noalloc"])
    if kind == "coupled":
        return dict(kind="coupled", config="c2", n=_log_int(rng, 257, 20000), periodic=rng.random() < 0.3)
    if kind == "steps":
        config = rng.choice(["c1", "c2", "c2", "n1e5"])
        n = _log_int(rng, 257, {"c1": 4096, "c2": 32768, "n1e5": 100000}[config])
        steps = min(20, max(1, int(MOST_PAIRS / n ** 2)))
        return dict(kind="steps", config=config, n=n, steps=steps, periodic=rng.random() < 0.3)
    if kind == "short":
        form = rng.choice(["delaunay", "delaunay", "verlet", "poly"])
        n = _log_int(rng, 3000, 50000 if form == "poly" else 700000)
        steps = min(20, max(1, int(MOST_DISK_STEPS / n)))
        case = dict(kind="steps", config="c3", n=n, steps=steps, periodic=rng.random() < 0.4)
        if form == "verlet":
            case["verlet"] = True
        if form == "poly":
            case["ratio"] = round(rng.uniform(1.1, 1.4), 3)
        return case
    if kind == "batch":
        return dict(kind="batch", replicas=rng.randint(8, 64), n_lo=512, n_hi=_log_int(rng, 2048, 16384),
                    steps=rng.randint(1, 4))
    if kind == "gradient":
        return dict(kind="gradient", config="c5", n=_log_int(rng, 500, 8192), steps=rng.randint(10, 40),
                    ckpt=rng.choice([7, 10, 20]), loss=rng.choice(["msd", "hist"]))
    if kind == "forces":
        return dict(kind="forces", config=rng.choice(["c1", "c2"]), n=_log_int(rng, 257, 30000),
                    periodic=rng.random() < 0.3)
    return dict(kind="noalloc", n=_log_int(rng, 257, 65536))


# ---------------------------------------------------------------- inputs

def _params(case, seed):
    cfg = CONFIG[case["config"]]
    p = bd.params_from_config(cfg, n=case["n"], seed=seed)
    p.box_L = workloads.box_side(case["n"], cfg.rho, cfg.a)
    if case.get("periodic"):
        p.boundary = bd.BOUNDARY_PERIODIC
    if case.get("verlet"):
        p.overlap_mode = bd.OVERLAP_VERLET
    return cfg, p


def _start(n, rho, a, n_species, seed):
    """Start positions as workloads.initial_state lays them out (random addition
    at low area fraction, the jittered lattice above), species, directions."""
    L = workloads.box_side(n, rho, a)
    xy = bd.place_disks(n, L, a, bd.PLACE_RSA if rho <= 0.35 else bd.PLACE_LATTICE, seed)
    rng = np.random.default_rng(seed)
    species = np.zeros(n, dtype=np.uint8)
    if n_species == 2:
        species[rng.permutation(n)[n // 2:]] = 1
    theta = rng.uniform(0.0, 2.0 * math.pi, size=n).astype(np.float32)
    return xy, species, theta


def _pinned(n):
    """Page-locked arrays that the state is read into and set from."""
    return (torch.empty((n, 2), dtype=torch.float64, pin_memory=True).numpy(),
            torch.empty((n,), dtype=torch.float32, pin_memory=True).numpy())


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        cfg = CONFIG["c2"]
        xy, sp, _ = _start(case["n"], cfg.rho, cfg.a, cfg.n_species, seed)
        n = case["n"]
        return dict(case=case, n=n, xy=torch.from_numpy(xy).cuda(), species=torch.from_numpy(sp).cuda(),
                    alpha=cfg.alpha, F=torch.empty((n, 2), dtype=torch.float64, device="cuda"))
    if kind == "batch":
        cfgs = workloads.batch_configs(case["replicas"], seed=3, n_lo=case["n_lo"], n_hi=case["n_hi"])
        plist, parts = [], []
        for r, cfg in enumerate(cfgs):
            p = bd.params_from_config(cfg, n=cfg.n, seed=seed)
            p.box_L = cfg.L
            p.replica = r
            plist.append(p)
            parts.append(_start(cfg.n, cfg.rho, cfg.a, cfg.n_species, 1000 * seed + r))
        xy, sp, th = (np.concatenate([q[k] for q in parts]) for k in range(3))
        system = bd.System(plist, xy, sp, th, stream=_stream())
        out_xy, out_th = _pinned(system.n)
        return dict(case=case, system=system, xy=out_xy, theta=out_th)
    cfg, p = _params(case, seed)
    xy, sp, th = _start(case["n"], cfg.rho, cfg.a, cfg.n_species, seed)
    radii = None
    if case.get("ratio"):
        radii = workloads.poly_radii(case["n"], cfg.a, case["ratio"], seed)
    system = bd.System(p, xy, sp, th, stream=_stream(), radii=radii)
    state = dict(case=case, system=system)
    if kind in ("steps", "coupled"):
        state["xy"], state["theta"] = _pinned(case["n"])
        system.read_state(state["xy"], state["theta"])
    if kind == "gradient":
        s = system.state(want_tri=False)
        state["xy0"], state["theta0"] = s["xy"], s["theta"]
        state["params"] = torch.tensor(list(cfg.alpha) + [cfg.v0], dtype=torch.float32)
    if kind == "forces":
        state["fp64"] = cfg.precision == 1
    return state


# ---------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "noalloc":
        binding.forces_noalloc(state["n"], state["xy"].data_ptr(), state["species"].data_ptr(), state["alpha"],
                          state["F"].data_ptr(), _stream())
        return state["F"].float()
    system = state["system"]
    if kind == "forces":
        F = system.forces()
        return F if state["fp64"] else F.astype(np.float32)
    if kind == "gradient":
        params = state["params"].clone().requires_grad_(True)
        loss = bd.rollout_loss(params, system, state["xy0"], state["theta0"], 0, case["steps"],
                               ckpt_every=case["ckpt"],
                               loss_kind=bd.LOSS_HIST if case["loss"] == "hist" else bd.LOSS_MSD)
        loss.backward()
        return {"loss": loss.detach().float(), "grad": params.grad}
    if kind == "coupled":
        system.set_state(state["xy"], state["theta"])
        system.step(1)
    else:
        system.step(case["steps"])
    system.read_state(state["xy"], state["theta"])
    return {"xy": state["xy"], "theta": state["theta"]}


# ---------------------------------------------------------------- work and exact values

def _step_work(n, law, precision):
    """One step: positions and directions read and written, the triangulation
    (two triangles a disk: corners and neighbours) read; the all-pairs law's 16
    flops per unordered pair, or about 8 pairs a disk of the short-range law."""
    b = n * (2 * (16 + 4) + 2 * 32)
    if law == workloads.LAW_LONG:
        return b, 16.0 * n * (n - 1) / 2
    return b, 8.0 * n * 60


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for cfg in workloads.batch_configs(case["replicas"], seed=3, n_lo=case["n_lo"], n_hi=case["n_hi"]):
            sb, sf = _step_work(cfg.n, cfg.law, cfg.precision)
            b += sb * case["steps"]
            f += sf * case["steps"]
        return {"bytes": b, "flops": f}
    n = case["n"]
    if kind in ("forces", "noalloc"):
        return {"bytes": n * (16 + 1 + 16), "flops": 16.0 * n * (n - 1) / 2}
    cfg = CONFIG[case["config"]]
    b, f = _step_work(n, cfg.law, cfg.precision)
    if kind == "gradient":
        # the steps, their replay, and the force adjoint (about 20 flops per ordered pair)
        return {"bytes": 3.0 * b * case["steps"], "flops": (2.0 * f + 20.0 * n * (n - 1)) * case["steps"]}
    return {"bytes": float(b * case.get("steps", 1)), "flops": float(f * case.get("steps", 1))}


def exact(case, seed):
    """The forces of the force cases as a plain FP64 sum over every pair.  The
    other cases' results depend on the discrete choices of a time step (flips,
    which pairs overlap) and have no plain closed form: None."""
    if case["kind"] not in ("forces", "noalloc"):
        return None
    cfg = CONFIG[case.get("config", "c2")]
    n = case["n"]
    xy, sp, _ = _start(n, cfg.rho, cfg.a, cfg.n_species, seed)
    x = torch.from_numpy(xy).cuda()
    s = torch.from_numpy(sp.astype(np.int64)).cuda()
    A = torch.tensor(cfg.alpha, dtype=torch.float64, device="cuda").reshape(2, 2)
    L = workloads.box_side(n, cfg.rho, cfg.a)
    L = float(np.float32(L)) if case.get("periodic") else None
    F = torch.empty_like(x)
    for i0 in range(0, n, 1024):
        r = x[i0:i0 + 1024, None, :] - x[None, :, :]
        if L is not None:
            r = r - L * torch.round(r / L)
        r2 = (r * r).sum(-1)
        c = A[s[i0:i0 + 1024]][:, s] * torch.where(r2 > 0, r2, torch.inf) ** -1.5
        F[i0:i0 + 1024] = (c[:, :, None] * r).sum(1)
    return F
