"""What a program that uses this package has it do, as cases that can be timed and checked.

Six tasks, each through the package's public entry points:

  md      relres_step on one system: molecular dynamics in calls of many steps (production runs) or of one
          step each (a program that looks at or changes the state between steps)
  frames  relres_compute on saved configurations of one system, forces only or with energies and virial;
          with ``rebuild`` every frame has its lists built anew (frames far apart in time)
  train   the differentiable form: energies, forces and the gradients of a force-matching loss with respect
          to positions and Lennard-Jones parameters, through torch.autograd
  batch   relres_batch_step: independent replicas of uneven sizes advanced together
  static  relres_pair_forces_static: the evaluation that allocates nothing, for small systems

over three liquids (propane-like, neopentane-like, block copolymer), the full FG reference (``fg_only``),
both precisions, NVE and thermostatted, and sizes from 648 atoms to the million-atom benchmark liquid.  A
system is a block of molecules repeated tx x ty x tz times, with seeded displacements of every molecule and
atom and seeded velocities, so that a large system costs no more to make than its arrays.

``exact`` evaluates the same quantities in 64 bits with plain torch (pair lists by cells, autograd for the
bonded terms and the gradients, velocity Verlet and the thermostat of Bussi, Donadio and Parrinello).
"""
import functools
import math

import numpy as np
import torch

from paper_2104_10231_gb300 import diff as D
from paper_2104_10231_gb300 import relres as R
from paper_2104_10231_gb300 import systems as S

TAU = 100.0        # thermostat time constant, fs
KB = 0.0019872042586408316
FTM2V = 4.184e-4   # (kcal/mol/A)/(g/mol) -> A/fs^2


# ------------------------------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest production run: the paper's 216-molecule propane box in double precision, NVE; a step
        # is a handful of short kernels, so latency and launches decide
        dict(name="md_propane_648_fp64", task="md", liquid="propane", block=6, tx=1, ty=1, tz=1, fp64=True,
             steps=100, calls=1, thermo=10, temp=0.0),
        # the everyday run: one thermostatted liquid of 20 000 atoms
        dict(name="md_neopentane_20k", task="md", liquid="neopentane", block=500, tx=2, ty=2, tz=2, fp64=False,
             steps=100, calls=1, thermo=50, temp=260.0),
        # the benchmark liquid: a million atoms, far larger than the caches
        dict(name="md_neopentane_1m", task="md", liquid="neopentane", block=1000, tx=5, ty=5, tz=8, fp64=False,
             steps=40, calls=1, thermo=20, temp=260.0),
        # polymers: dihedrals, four types, excluded pairs inside long chains, chain segments
        dict(name="md_copolymer_14k", task="md", liquid="copolymer", block=12, tx=2, ty=2, tz=3, fp64=False,
             steps=50, calls=1, thermo=25, temp=300.0),
        # a reference trajectory in double precision at a production size
        dict(name="md_neopentane_25k_fp64", task="md", liquid="neopentane", block=1000, tx=1, ty=1, tz=5, fp64=True,
             steps=40, calls=1, thermo=20, temp=260.0),
        # a program that drives the run step by step (biasing, coupling to another code): one step per call
        dict(name="single_steps_propane_140k", task="md", liquid="propane", block=9, tx=4, ty=4, tz=4, fp64=False,
             steps=1, calls=8, thermo=0, temp=230.0),
        # the smallest evaluation: forces of a small system, one configuration after another
        dict(name="frames_propane_1k", task="frames", liquid="propane", block=7, tx=1, ty=1, tz=1, fp64=False,
             frames=8, energy=False, rebuild=False, fg_only=False),
        # energies, virial and forces of saved configurations at the everyday size
        dict(name="frames_neopentane_20k", task="frames", liquid="neopentane", block=500, tx=2, ty=2, tz=2,
             fp64=False, frames=8, energy=True, rebuild=False, fg_only=False),
        # scoring far-apart frames with the full FG reference the method is compared with: lists from
        # scratch, then long list walks with energies
        dict(name="rescore_fg_only_250k", task="frames", liquid="neopentane", block=1000, tx=5, ty=5, tz=2,
             fp64=False, frames=2, energy=True, rebuild=True, fg_only=True),
        # fitting the parameters by force matching: forward and backward per snapshot
        dict(name="train_neopentane_20k", task="train", liquid="neopentane", block=500, tx=2, ty=2, tz=2,
             fp64=False, frames=4),
        # a set of replicas of uneven sizes, alternately propane- and neopentane-like
        dict(name="batch_mixed_24", task="batch", replicas=24, least=1000, most=30000, shape=1, steps=25, thermo=25),
        # the no-allocation evaluation of a host program's small system, with exclusions, energy and virial
        dict(name="static_propane_4k", task="static", liquid="propane", block=11, tx=1, ty=1, tz=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _tiles(rng, count):
    """Three factors whose product is near `count`."""
    a = max(1, min(12, int(round(count ** (1 / 3) * math.exp(rng.uniform(-0.3, 0.3))))))
    b = max(1, min(12, int(round(math.sqrt(count / a) * math.exp(rng.uniform(-0.2, 0.2))))))
    c = max(1, min(16, int(round(count / (a * b)))))
    t = [a, b, c]
    rng.shuffle(t)
    return t


def _lattice(n):
    """A number of molecules near n that a cubic lattice holds without crowding: 85 to 100 % of its sites."""
    k = max(7, math.ceil(n ** (1 / 3) - 1e-9))
    return int(min(k ** 3, max(math.ceil(0.85 * k ** 3), round(n))))


def _draw_system(rng, liquid, lo, hi):
    n = _log_int(rng, lo, hi)
    if liquid == "propane":
        # blocks of k^3 molecules; at least 648 atoms, so that 14 A fits half the box
        k = rng.randint(6, 11)
        per = 3 * k ** 3
    elif liquid == "neopentane":
        k = _lattice(rng.uniform(300, 1000))
        per = 5 * k
    else:
        k = rng.choice([12, 13])
        per = 100 * k
    tx, ty, tz = _tiles(rng, max(1.0, n / per))
    while per * tx * ty * tz > hi and max(tx, ty, tz) > 1:  # never above the range
        t = sorted([tx, ty, tz])
        tx, ty, tz = t[0], t[1], t[2] - 1
    return dict(liquid=liquid, block=k, tx=tx, ty=ty, tz=tz)


def draw(rng):
    task = rng.choices(["md", "frames", "train", "batch", "static"], [5, 3, 2, 1, 1])[0]
    if task == "md":
        fp64 = rng.random() < 0.3
        liquid = rng.choice(["propane", "neopentane", "neopentane", "copolymer"])
        hi = {"copolymer": 20000, "propane": 30000, "neopentane": 30000}[liquid] if fp64 else \
            {"copolymer": 40000, "propane": 400000, "neopentane": 900000}[liquid]
        c = dict(task="md", **_draw_system(rng, liquid, 648, hi), fp64=fp64)
        n = _atoms(c)
        one = rng.random() < 0.25
        steps = 1 if one else rng.randint(20, max(21, min(100, 12_000_000 // n)))
        c.update(steps=steps, calls=rng.randint(3, 8) if one else 1, thermo=0 if one else rng.choice([0, 7, 10]),
                 temp=rng.choice([0.0, round(rng.uniform(200.0, 300.0), 1)]))
        return c
    if task == "frames":
        fp64 = rng.random() < 0.3
        liquid = rng.choice(["propane", "neopentane", "copolymer"])
        hi = 20000 if fp64 else {"copolymer": 20000}.get(liquid, 250000)
        c = dict(task="frames", **_draw_system(rng, liquid, 648, hi), fp64=fp64)
        c.update(frames=rng.randint(1, 8) if _atoms(c) < 60000 else rng.randint(1, 2), energy=rng.random() < 0.6,
                 rebuild=rng.random() < 0.3, fg_only=liquid == "neopentane" and rng.random() < 0.3)
        return c
    if task == "train":
        fp64 = rng.random() < 0.3
        liquid = rng.choice(["propane", "neopentane", "copolymer"])
        c = dict(task="train", **_draw_system(rng, liquid, 648, 8000 if fp64 else 40000), fp64=fp64)
        c.update(frames=rng.randint(1, 4))
        return c
    if task == "batch":
        least = _log_int(rng, 700, 4000)
        return dict(task="batch", replicas=rng.randint(5, 24), least=least, most=_log_int(rng, least + 200, 30000),
                    shape=rng.randint(2, 1 << 20), steps=rng.randint(10, 25), thermo=rng.choice([0, 5]))
    return dict(task="static", liquid="propane", block=rng.randint(6, 12), tx=1, ty=1, tz=1)


# ------------------------------------------------------------------------------------------- systems

def _atoms(case):
    per = {"propane": 3 * case["block"] ** 3, "neopentane": 5 * case["block"], "copolymer": 100 * case["block"]}
    return per[case["liquid"]] * case["tx"] * case["ty"] * case["tz"]


@functools.lru_cache(maxsize=40)
def _block(liquid, block):
    if liquid == "propane":
        return S.propane(n_mol=block ** 3, box=31.8 * block / 6)
    if liquid == "neopentane":
        return S.neopentane(n_mol=block)
    return _relaxed(S.block_copolymer(n_chain=block))


def _relaxed(s, rounds=8):
    """Chains grown at random start with stretched contacts: downhill by at most 0.05 A a step, on the host, so
    that every process gets the same block."""
    field = _Field(s, dev="cpu")
    x = torch.tensor(s.pos)
    for _ in range(rounds):
        lists = field.lists(x, 2.0)
        for _ in range(20):
            x = x + torch.clamp(5e-4 * field.all(x, lists)[3], -0.05, 0.05)
    return s.subset_copy(pos=(x - torch.floor(x / field.box) * field.box).numpy())


@functools.lru_cache(maxsize=40)
def _system(liquid, block, tx, ty, tz):
    """The block repeated tx x ty x tz times (host arrays: the topology a program reads from its files)."""
    b = _block(liquid, block)
    nt, n = tx * ty * tz, b.n_atoms
    if nt == 1:
        return b
    off = np.stack(np.meshgrid(np.arange(tx), np.arange(ty), np.arange(tz), indexing="ij"), -1).reshape(-1, 3)
    # whole molecules: an atom beside its predecessor, not across the block's own boundary
    step = np.diff(b.pos, axis=0)
    step -= np.round(step / b.box) * b.box
    first = np.concatenate([[True], np.diff(b.mol) != 0])
    step = np.concatenate([np.zeros((1, 3)), step])
    walked = np.cumsum(step, axis=0)
    head = np.maximum.accumulate(np.where(first, np.arange(n), 0))
    pos = b.pos[head] + walked - walked[head]
    pos = (pos[None] + (off * b.box)[:, None, :]).reshape(-1, 3)
    shift = (np.arange(nt) * n).astype(np.int32)

    def moved(idx, width):
        return (idx.reshape(1, -1, width) + shift[:, None, None]).reshape(-1, width).astype(np.int32)

    topo = dict(b.topo)
    for key, width in (("bonds", 2), ("angles", 3), ("dihedrals", 4)):
        topo[key] = moved(np.asarray(b.topo[key]), width)
    for key in ("bond_type", "angle_type", "dihedral_type"):
        topo[key] = np.tile(b.topo[key], nt)
    ei = (b.excl_idx[None, :] + shift[:, None]).reshape(-1).astype(np.int32)
    eo = np.concatenate([(b.excl_off[None, :-1] + (np.arange(nt) * len(b.excl_idx))[:, None]).reshape(-1),
                         [nt * len(b.excl_idx)]]).astype(np.int32)
    n_mol = int(b.mol.max()) + 1
    mol = (b.mol[None] + (np.arange(nt) * n_mol)[:, None]).reshape(-1).astype(np.int32)
    return b.subset_copy(pos=pos, vel=np.zeros_like(pos), types=np.tile(b.types, nt), mol=mol,
                         box=b.box * np.array([tx, ty, tz]), topo=topo, excl_off=eo, excl_idx=ei)


def _sys(case):
    s = _system(case["liquid"], case["block"], case["tx"], case["ty"], case["tz"])
    return S.fg_only(s) if case.get("fg_only") else s


@functools.lru_cache(maxsize=40)
def _on_gpu(liquid, block, tx, ty, tz):
    s = _system(liquid, block, tx, ty, tz)
    return (torch.tensor(s.pos, device="cuda"), torch.tensor(s.mol, device="cuda").long(),
            torch.tensor(s.masses, device="cuda"))


def _start(case, seed, per_atom, temp):
    """Seeded positions (every molecule and atom displaced) and Maxwell-Boltzmann velocities."""
    base, mol, mass = _on_gpu(case["liquid"], case["block"], case["tx"], case["ty"], case["tz"])
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 13)

    def normal(n):
        return torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)

    box = torch.tensor(_sys(case).box, device="cuda")
    shift = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * box
    pos = base + shift + 0.05 * normal(int(mol[-1]) + 1)[mol] + per_atom * normal(len(base))
    pos = pos - torch.floor(pos / box) * box
    vel = normal(len(base)) * torch.sqrt(KB * (temp or 230.0) / mass * FTM2V)[:, None]
    vel = vel - (vel * mass[:, None]).sum(0) / mass.sum()
    return pos, vel, g


def _precision(case):
    return R.RELRES_PREC_FP64 if case.get("fp64") else R.RELRES_PREC_FP32


def _dt(case):
    return 2.0 if case["liquid"] == "neopentane" else 1.0


@functools.lru_cache(maxsize=40)
def _marshalled(liquid, block, tx, ty, tz, fp64, fg_only):
    s = _system(liquid, block, tx, ty, tz)
    s = S.fg_only(s) if fg_only else s
    return R.params_for(s, R.RELRES_PREC_FP64 if fp64 else R.RELRES_PREC_FP32), R.topology_for(s)


def _context(case, pos):
    p, t = _marshalled(case["liquid"], case["block"], case["tx"], case["ty"], case["tz"], bool(case.get("fp64")),
                       bool(case.get("fg_only")))
    ctx = R.Context(p, t)
    ctx.build_neighbors(pos, _sys(case).box)
    return ctx


def _frames(case, seed, per_atom):
    """Saved configurations: one start, every frame with its own noise (per_atom A per coordinate)."""
    base, _, g = _start(case, seed, 0.02, 0.0)
    n = len(base)
    noise = torch.randn(case["frames"], n, 3, generator=g, device="cuda", dtype=torch.float64)
    return base, base + per_atom * noise


# a set of replicas: sizes drawn once from `shape`, alternately propane- and neopentane-like
def _replicas(case):
    rng = np.random.default_rng(case["shape"])
    out = []
    for k in range(case["replicas"]):
        n = math.exp(rng.uniform(math.log(case["least"]), math.log(case["most"])))
        if k % 2 == 0:
            m = max(6, int(round((n / 3) ** (1 / 3))))
            one = dict(liquid="propane", block=m, tx=1, ty=1, tz=1)
        else:
            parts = max(1, math.ceil(n / 5000))
            one = dict(liquid="neopentane", block=_lattice(n / 5 / parts), tx=1, ty=1, tz=parts)
        one["temp"] = round(float(rng.uniform(200.0, 300.0)), 1)
        out.append(one)
    return out


class _BatchState(dict):
    """Closes the batch before its contexts go."""

    def __del__(self):
        try:
            self["batch"].close()
        except Exception:
            pass


def _noise_of(case):
    # small displacements where the frames also stretch bonds, the thermal ones where only pairs count
    return 0.15 if case["task"] == "train" else 0.1


# ------------------------------------------------------------------------------------------- prepare, run

def prepare(case, seed):
    task = case["task"]
    if task == "md":
        pos, vel, _ = _start(case, seed, 0.02, case["temp"])
        ctx = _context(case, pos)
        rows = case["steps"] // case["thermo"] if case["thermo"] else 0
        thermo = torch.zeros(max(1, rows), R.RELRES_THERMO_COLS, dtype=torch.float64, device="cuda") if rows else None
        return dict(case=case, ctx=ctx, pos=pos, vel=vel, thermo=thermo, seed=seed % 1000003, dt=_dt(case))
    if task == "frames":
        base, frames = _frames(case, seed, _noise_of(case))
        ctx = _context(case, base)
        k, n = frames.shape[:2]
        return dict(case=case, ctx=ctx, frames=frames, box=_sys(case).box, forces=torch.empty_like(frames),
                    energy=torch.zeros(k, 4, dtype=torch.float64, device="cuda"),
                    virial=torch.zeros(k, 6, dtype=torch.float64, device="cuda"))
    if task == "train":
        s = _sys(case)
        base, frames = _frames(case, seed, _noise_of(case))
        model = D.RelResPair.for_system(s, _precision(case))
        model.bind(base, s.box)
        eps = torch.tensor(s.eps_fg * 1.03, requires_grad=True)
        sig = torch.tensor(s.sig_fg * 0.995, requires_grad=True)
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
        ref = 2.0 * torch.randn(frames.shape, generator=g, device="cuda", dtype=torch.float64)
        return dict(case=case, model=model, frames=[f.clone().requires_grad_(True) for f in frames], ref=ref,
                    eps=eps, sig=sig)
    if task == "batch":
        reps = _replicas(case)
        starts = [_start(r, seed * 64 + k, 0.02, r["temp"]) for k, r in enumerate(reps)]
        sizes = [len(p) for p, _, _ in starts]
        pos, vel = torch.cat([p for p, _, _ in starts]), torch.cat([v for _, v, _ in starts])
        rows = case["steps"] // case["thermo"] if case["thermo"] else 0
        thermo = torch.zeros(len(reps), rows, R.RELRES_THERMO_COLS, dtype=torch.float64, device="cuda") if rows else None
        ps, vs = list(pos.split(sizes)), list(vel.split(sizes))
        ctxs = [_context(r, p) for r, p in zip(reps, ps)]
        return _BatchState(case=case, ctxs=ctxs, batch=R.Batch(ctxs), pos=pos, vel=vel, ps=ps, vs=vs, thermo=thermo,
                           th=list(thermo) if rows else None, temps=[r["temp"] for r in reps],
                           seeds=[seed % 1000003 + k for k in range(len(reps))])
    s = _sys(case)
    pos, _, _ = _start(case, seed, 0.1, 0.0)
    return dict(case=case, params=R.params_for(s, R.RELRES_PREC_FP64), box=s.box, n=s.n_atoms, pos=pos,
                types=torch.tensor(s.types, device="cuda"), eo=torch.tensor(s.excl_off, device="cuda"),
                ei=torch.tensor(s.excl_idx, device="cuda"), forces=torch.empty_like(pos),
                energy=torch.zeros(1, dtype=torch.float64, device="cuda"),
                virial=torch.zeros(6, dtype=torch.float64, device="cuda"))


def run(state):
    case = state["case"]
    task = case["task"]
    if task == "md":
        for _ in range(case["calls"]):
            state["ctx"].step(case["steps"], state["dt"], state["pos"], state["vel"], t_target=case["temp"],
                              tau_fs=TAU, seed=state["seed"], thermo_every=case["thermo"], d_thermo=state["thermo"])
        out = dict(pos=state["pos"], vel=state["vel"])
        if state["thermo"] is not None:
            out["thermo"] = state["thermo"]
        return out
    if task == "frames":
        e = case["energy"]
        for k in range(case["frames"]):
            if case["rebuild"]:
                state["ctx"].build_neighbors(state["frames"][k], state["box"])
            state["ctx"].compute(state["frames"][k], state["forces"][k], state["energy"][k] if e else None,
                                 state["virial"][k] if e else None)
        out = dict(forces=state["forces"])
        if e:
            out.update(energy=state["energy"], virial=state["virial"])
        return out
    if task == "train":
        eps, sig = state["eps"], state["sig"]
        eps.grad = sig.grad = None
        energies = []
        for k, x in enumerate(state["frames"]):
            x.grad = None
            e, f = state["model"](x, eps, sig)
            loss = 0.001 * e + ((f - state["ref"][k]) ** 2).sum() / f.numel()
            loss.backward()
            energies.append(e.detach())
            last = f.detach()
        return dict(energy=torch.stack(energies), last_forces=last, grad_pos=[x.grad for x in state["frames"]],
                    grad_eps=eps.grad, grad_sig=sig.grad)
    if task == "batch":
        state["batch"].step(case["steps"], 1.0, state["ps"], state["vs"], state["temps"], TAU, state["seeds"],
                            case["thermo"], state["th"])
        out = dict(pos=state["pos"], vel=state["vel"])
        if state["thermo"] is not None:
            out["thermo"] = state["thermo"]
        return out
    R.relres_pair_forces_static(state["params"], state["n"], state["types"], state["pos"], state["box"],
                                state["forces"], state["energy"], state["virial"], state["eo"], state["ei"])
    return dict(forces=state["forces"], energy=state["energy"], virial=state["virial"])


# ------------------------------------------------------------------------------------------- work, tolerance

def _pairs(s):
    """FG and CG pairs inside the interaction ranges (each once), at the liquid's uniform density."""
    vol = float(np.prod(s.box))
    n, nh = s.n_atoms, s.n_hybrid
    fg = 0.5 * n * n * 4.18879 * s.radii[1] ** 3 / vol
    cg = 0.5 * nh * nh * 4.18879 * s.radii[3] ** 3 / vol
    return fg, cg


def work(case):
    """Each input read once and each output written once per pass (positions, velocities, forces: 24 bytes an
    atom each), and the arithmetic of the interacting pairs, each once: about 45 operations for a force, 30 more
    for its energy and virial, 3 times that for second derivatives."""
    task = case["task"]
    if task == "batch":
        f = b = 0.0
        for r in _replicas(case):
            s = _sys(r)
            f += case["steps"] * (45.0 * sum(_pairs(s)) + 100.0 * s.n_atoms)
            b += 96.0 * s.n_atoms
        return dict(bytes=b, flops=f)
    s = _sys(case)
    n, pairs = s.n_atoms, sum(_pairs(s))
    if task == "md":
        k = case["steps"] * case["calls"]
        return dict(bytes=96.0 * n * case["calls"], flops=k * (45.0 * pairs + 100.0 * n))
    if task == "frames":
        return dict(bytes=48.0 * n * case["frames"], flops=case["frames"] * pairs * (75.0 if case["energy"] else 45.0))
    if task == "train":
        return dict(bytes=(48.0 + 72.0) * n * case["frames"], flops=case["frames"] * pairs * (75.0 + 135.0))
    return dict(bytes=(48.0 + 4.0) * n, flops=75.0 * pairs)


def tolerance(case):
    """Four times what was seen against `exact`, and between force sums in another order or precision, over the
    listed cases and ten drawn ones.  Double precision: up to 8e-13 (energies and virial whose parts cancel, with
    the trajectories' own growth on top).  Single precision: forces 1e-7, virials 9e-7, velocities after up to 200
    steps 8e-7; gradients that hold second derivatives of close pairs 2.5e-6."""
    if case["task"] == "static" or case.get("fp64"):
        return {"rel": 4e-12, "max": 4e-10}
    if case["task"] == "train":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 4e-6, "max": 1e-4}


# ------------------------------------------------------------------------------------------- exact

def _pair_list(pos, box, cut, sel=None, excl=None):
    """All pairs (i < j in slot order) of the atoms `sel` closer than `cut` (minimum image), without `excl`."""
    n_all = len(pos)
    x = pos if sel is None else pos[sel]
    x = x - torch.floor(x / box) * box
    n = len(x)
    nc = [int(v) for v in torch.clamp(torch.floor(box / cut), min=1, max=400).tolist()]
    got = []

    def keep(i, j):
        d = x[i] - x[j]
        d = d - torch.round(d / box) * box
        ok = (d * d).sum(1) < cut * cut
        got.append((i[ok], j[ok]))

    if min(nc) < 3:
        step = max(1, 20_000_000 // n)
        ar = torch.arange(n, device=x.device)
        for lo in range(0, n, step):
            i = ar[lo:lo + step]
            m = i[:, None] < ar[None, :]
            a, b = m.nonzero(as_tuple=True)
            keep(i[a], ar[b])
    else:
        nct = torch.tensor(nc, device=x.device)
        c3 = torch.minimum(torch.floor(x / box * nct).long(), nct - 1)
        cell = (c3[:, 0] * nc[1] + c3[:, 1]) * nc[2] + c3[:, 2]
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=nc[0] * nc[1] * nc[2])
        start = torch.cumsum(count, 0) - count
        offs = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if (a, b, c) >= (0, 0, 0)]
        for o in offs:
            c2 = torch.remainder(c3 + torch.tensor(o, device=x.device), nct)
            cc = (c2[:, 0] * nc[1] + c2[:, 1]) * nc[2] + c2[:, 2]
            step = max(1, 30_000_000 // max(1, int(count.max())))
            for lo in range(0, n, step):
                i = torch.arange(lo, min(n, lo + step), device=x.device)
                k = count[cc[i]]
                a = torch.repeat_interleave(i, k)
                first = torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
                b = order[torch.repeat_interleave(start[cc[i]], k) + torch.arange(len(a), device=x.device) - first]
                if o == (0, 0, 0):
                    m = a < b
                    a, b = a[m], b[m]
                keep(a, b)
    i, j = torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    if sel is not None:
        i, j = sel[i], sel[j]
    if excl is not None and len(excl):
        key = i * n_all + j
        at = torch.clamp(torch.searchsorted(excl, key), max=len(excl) - 1)
        m = excl[at] != key
        i, j = i[m], j[m]
    return i, j


def _poly_off(u, du, d2u, w):
    return [u, du, 0.5 * d2u, -(du / w ** 2) - 2 * d2u / (3 * w), du / (2 * w ** 3) + d2u / (4 * w ** 2)]


def _poly_on(u, du, d2u, w):
    z = torch.zeros_like(u)
    return [u - 0.5 * du * w + d2u * w * w / 12, z, z, du / w ** 2 - d2u / (3 * w), d2u / (4 * w * w) - du / (2 * w ** 3)]


def _poly(g, d):
    return (((g[4] * d + g[3]) * d + g[2]) * d + g[1]) * d + g[0]


class _Field:
    """The pair potential and bonded terms of one system in 64 bits (the paper's Eq. 11-20)."""

    def __init__(self, s, eps=None, sig=None, dev="cuda"):
        self.s, self.dev = s, dev
        self.box = torch.tensor(s.box, device=dev)
        self.types = torch.tensor(s.types, device=dev).long()
        self.rsm, self.rsp, self.rcm, self.rcp = s.radii
        hyb = torch.tensor(s.is_hybrid, device=dev).bool()
        self.sel = hyb[self.types].nonzero()[:, 0]
        cnt = torch.tensor(np.diff(s.excl_off), device=dev).long()
        i = torch.repeat_interleave(torch.arange(s.n_atoms, device=dev), cnt)
        self.excl = torch.sort(i * s.n_atoms + torch.tensor(s.excl_idx, device=dev).long())[0]
        self.set(torch.tensor(s.eps_fg, device=dev) if eps is None else eps,
                 torch.tensor(s.sig_fg, device=dev) if sig is None else sig)
        t = s.topo
        self.bonded = {k: torch.tensor(np.asarray(t[k]), device=dev) for k in t}

    def set(self, eps, sig):
        s, dev = self.s, self.dev
        e = torch.sqrt(eps[:, None] * eps[None, :])
        r = 0.5 * (sig[:, None] + sig[None, :]) if s.mixing == "lb" else torch.sqrt(sig[:, None] * sig[None, :])
        comp = torch.tensor(s.group_comp, device=dev).double()
        hh = torch.tensor(np.outer(s.is_hybrid, s.is_hybrid), device=dev).bool()
        a6, a12 = comp @ (e * r ** 6) @ comp.T, comp @ (e * r ** 12) @ comp.T
        one = torch.ones_like(a6)
        a6, a12 = torch.where(hh, a6, one), torch.where(hh, a12, one)
        z = torch.zeros_like(a6)
        # 4 eps sig^12, 4 eps sig^6: the CG pair has eps sig^6 = A6 and eps sig^12 = A12 (Eq. 4)
        self.f = (4 * e * r ** 12, 4 * e * r ** 6)
        self.c = (torch.where(hh, 4 * a12, z), torch.where(hh, 4 * a6, z))
        w, wc = self.rsp - self.rsm, self.rcp - self.rcm
        self.g_off = _poly_off(*self._lj3(self.f, self.rsm), w)
        self.sh = _poly(self.g_off, w)
        self.has_cg = bool(hh.any())
        if self.has_cg:
            self.g_on = _poly_on(*self._lj3(self.c, self.rsp), w)
            self.g_cut = _poly_off(*self._lj3(self.c, self.rcm), wc)
            self.gam = _poly(self.g_cut, wc)

    @staticmethod
    def _lj3(c, r):
        return (c[0] * r ** -12 - c[1] * r ** -6, -12 * c[0] * r ** -13 + 6 * c[1] * r ** -7,
                156 * c[0] * r ** -14 - 42 * c[1] * r ** -8)

    def lists(self, pos, skin):
        fg = _pair_list(pos, self.box, self.rsp + skin, None, self.excl)
        cg = _pair_list(pos, self.box, self.rcp + skin, self.sel, self.excl) if self.has_cg else None
        return fg, cg

    def _lj(self, c, k, r2):
        i6 = 1.0 / (r2 * r2 * r2)
        return (c[0].reshape(-1)[k] * i6 - c[1].reshape(-1)[k]) * i6

    def u_fg(self, r, k):
        t = [g.reshape(-1)[k] for g in self.g_off]
        inner = r < self.rsm
        u = torch.where(inner, self._lj(self.f, k, torch.where(inner, r, self.rsm) ** 2), _poly(t, r - self.rsm))
        return u - self.sh.reshape(-1)[k]

    def u_cg(self, r, k):
        on, cut = [g.reshape(-1)[k] for g in self.g_on], [g.reshape(-1)[k] for g in self.g_cut]
        u = torch.where(r < self.rsp, _poly(on, torch.clamp(r - self.rsm, min=0.0)),
                        torch.where(r < self.rcm, self._lj(self.c, k, torch.clamp(r, min=self.rsp) ** 2),
                                    _poly(cut, r - self.rcm)))
        return u - self.gam.reshape(-1)[k]

    def pairs(self, pos, lists, graph=False):
        """E_fg, E_cg, forces, virial of the pairs; graph: everything stays differentiable."""
        n = len(pos)
        f = torch.zeros_like(pos)
        w = torch.zeros(6, dtype=pos.dtype, device=pos.device)
        es = []
        for lst, cut, u in ((lists[0], self.rsp, self.u_fg), (lists[1], self.rcp, self.u_cg)):
            if lst is None:
                es.append(torch.zeros((), dtype=pos.dtype, device=pos.device))
                continue
            i, j = lst
            with torch.no_grad():
                d = pos[i] - pos[j]
                im = torch.round(d / self.box) * self.box
                ok = ((d - im) ** 2).sum(1) < cut * cut
            i, j, im = i[ok], j[ok], im[ok]
            d = pos[i] - pos[j] - im
            r = torch.sqrt((d * d).sum(1))
            if not graph:
                r = r.detach().requires_grad_(True)
            with torch.enable_grad():
                e = u(r, self.types[i] * self.s.n_types + self.types[j])
                du, = torch.autograd.grad(e.sum(), r, create_graph=graph)
            if not graph:
                e, r = e.detach(), r.detach()
            fd = (-du / r)[:, None] * d
            f = f.index_add(0, i, fd).index_add(0, j, -fd)
            w = w + torch.stack([(d[:, a] * fd[:, b]).sum() for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
            es.append(e.sum())
        return es[0], es[1], f, w

    def bonded_energy(self, pos):
        t = self.bonded

        def diff(a, b):
            d = pos[a] - pos[b]
            return d - torch.round(d.detach() / self.box) * self.box

        e = torch.zeros((), dtype=pos.dtype, device=pos.device)
        if len(t["bond_type"]):
            b, k = t["bonds"].long(), t["bond_type"].long()
            r = torch.sqrt((diff(b[:, 0], b[:, 1]) ** 2).sum(1))
            e = e + (t["bond_k"][k] * (r - t["bond_r0"][k]) ** 2).sum()
        if len(t["angle_type"]):
            a, k = t["angles"].long(), t["angle_type"].long()
            p, q = diff(a[:, 0], a[:, 1]), diff(a[:, 2], a[:, 1])
            th = torch.atan2(torch.sqrt((torch.linalg.cross(p, q) ** 2).sum(1)), (p * q).sum(1))
            e = e + (t["angle_k"][k] * (th - t["angle_theta0"][k]) ** 2).sum()
        if len(t["dihedral_type"]):
            a, k = t["dihedrals"].long(), t["dihedral_type"].long()
            b1, b2, b3 = diff(a[:, 1], a[:, 0]), diff(a[:, 2], a[:, 1]), diff(a[:, 3], a[:, 2])
            m1, m2 = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
            phi = torch.atan2(torch.sqrt((b2 * b2).sum(1)) * (b1 * m2).sum(1), (m1 * m2).sum(1))
            kk = t["dihedral_k"][k]
            e = e + 0.5 * (kk[:, 0] * (1 + torch.cos(phi)) + kk[:, 1] * (1 - torch.cos(2 * phi))
                           + kk[:, 2] * (1 + torch.cos(3 * phi)) + kk[:, 3] * (1 - torch.cos(4 * phi))).sum()
        return e

    def all(self, pos, lists):
        ef, ec, f, w = self.pairs(pos, lists)
        if any(len(self.bonded[k]) for k in ("bond_type", "angle_type", "dihedral_type")):
            x = pos.detach().requires_grad_(True)
            with torch.enable_grad():
                eb = self.bonded_energy(x)
                g, = torch.autograd.grad(eb, x)
            return ef, ec, eb.detach(), f - g, w
        return ef, ec, torch.zeros_like(ef), f, w


# the thermostat's random numbers: splitmix64 read at a counter, Box-Muller, Marsaglia and Tsang
_M64 = (1 << 64) - 1


class _Draws:
    def __init__(self, key, step):
        self.key, self.c = key, step << 20

    def uniform(self):
        self.c += 1
        z = (self.key + self.c * 0x9E3779B97F4A7C15) & _M64
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
        return (float((z ^ (z >> 31)) >> 11) + 1.0) * 2.0 ** -53

    def normal(self):
        a, b = self.uniform(), self.uniform()
        return math.sqrt(-2.0 * math.log(a)) * math.cos(2.0 * math.pi * b)

    def gamma(self, shape):
        d = shape - 1.0 / 3.0
        k = 1.0 / math.sqrt(9.0 * d)
        while True:
            x = self.normal()
            v = 1.0 + k * x
            if v <= 0.0:
                continue
            v = v ** 3
            if math.log(self.uniform()) < 0.5 * x * x + d - d * v + d * math.log(v):
                return d * v


def _exact_md(s, pos, vel, steps, dt, temp, seed, thermo_every):
    field = _Field(s)
    m = torch.tensor(s.masses, device=pos.device)[:, None]
    x, v = pos.clone(), vel.clone()
    ref, lists = x, field.lists(x, 2.0)
    f = field.all(x, lists)[3]
    n_f = 3.0 * len(x) - 3.0
    rows = []
    for k in range(steps):
        v = v + 0.5 * dt * FTM2V * f / m
        x = x + dt * v
        if float(((x - ref) ** 2).sum(1).max()) > 0.98:
            ref, lists = x, field.lists(x, 2.0)
        ef, ec, eb, f, w = field.all(x, lists)
        v = v + 0.5 * dt * FTM2V * f / m
        ke = float((m * v * v).sum()) * 0.5 / FTM2V
        if temp > 0.0:
            d = _Draws(seed, k)
            r1 = d.normal()
            chi = 2.0 * d.gamma(0.5 * (n_f - 1.0))
            c, kt = math.exp(-dt / TAU), 0.5 * n_f * KB * temp
            kn = ke + (1 - c) * (kt / n_f * (r1 * r1 + chi) - ke) + 2 * r1 * math.sqrt(c * (1 - c) * ke * kt / n_f)
            v = v * math.sqrt(kn / ke)
            ke = kn
        if thermo_every and (k + 1) % thermo_every == 0:
            rows.append(torch.cat([torch.stack([ef, ec, eb, torch.tensor(ke, device=pos.device, dtype=pos.dtype)]), w]))
    out = dict(pos=x - torch.floor(x / field.box) * field.box, vel=v)
    if rows:
        out["thermo"] = torch.stack(rows)
    return out


def exact(case, seed):
    task = case["task"]
    if task == "md":
        pos, vel, _ = _start(case, seed, 0.02, case["temp"])
        return _exact_md(_sys(case), pos, vel, case["steps"] * case["calls"], _dt(case), case["temp"], seed % 1000003,
                         case["thermo"])
    if task == "batch":
        got = []
        for k, r in enumerate(_replicas(case)):
            pos, vel, _ = _start(r, seed * 64 + k, 0.02, r["temp"])
            got.append(_exact_md(_sys(r), pos, vel, case["steps"], 1.0, r["temp"], seed % 1000003 + k, case["thermo"]))
        out = dict(pos=torch.cat([g["pos"] for g in got]), vel=torch.cat([g["vel"] for g in got]))
        if case["thermo"]:
            out["thermo"] = torch.stack([g["thermo"] for g in got])
        return out
    if task == "frames":
        s = _sys(case)
        _, frames = _frames(case, seed, _noise_of(case))
        field = _Field(s)
        got = [field.all(x, field.lists(x, 0.0)) for x in frames]
        out = dict(forces=torch.stack([g[3] for g in got]))
        if case["energy"]:
            out["energy"] = torch.stack([torch.stack([g[0], g[1], g[2], g[0] + g[1] + g[2]]) for g in got])
            out["virial"] = torch.stack([g[4] for g in got])
        return out
    if task == "train":
        s = _sys(case)
        _, frames = _frames(case, seed, _noise_of(case))
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
        ref = 2.0 * torch.randn(frames.shape, generator=g, device="cuda", dtype=torch.float64)
        eps = torch.tensor(s.eps_fg * 1.03, device="cuda", requires_grad=True)
        sig = torch.tensor(s.sig_fg * 0.995, device="cuda", requires_grad=True)
        energies, grads = [], []
        for x, r in zip(frames, ref):
            x = x.clone().requires_grad_(True)
            field = _Field(s, eps, sig)
            ef, ec, f, _ = field.pairs(x, field.lists(x.detach(), 0.0), graph=True)
            (0.001 * (ef + ec) + ((f - r) ** 2).sum() / f.numel()).backward()
            energies.append((ef + ec).detach())
            grads.append(x.grad)
        return dict(energy=torch.stack(energies), last_forces=f.detach(), grad_pos=grads, grad_eps=eps.grad,
                    grad_sig=sig.grad)
    s = _sys(case)
    pos, _, _ = _start(case, seed, 0.1, 0.0)
    field = _Field(s)
    ef, ec, f, w = field.pairs(pos, field.lists(pos, 0.0))
    return dict(forces=f, energy=(ef + ec).reshape(1), virial=w)
