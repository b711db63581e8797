"""FP32 pair launches with several lanes per list (systems too small to fill the
GPU with one thread per list) and the FP32 energy steps: the force bits of one
thread per list, energies and virial that do not depend on the launch, and
pruned lists with the same entries in the same order."""
import numpy as np
import pytest

from paper_2104_10231_gb300 import relres as R
from paper_2104_10231_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as T

    assert T.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2104_10231_gb300.build import build_library

    build_library()
    R.load()
    return T


def _dev(torch, a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


# list owners (atoms + hybrids) around the changes of the rule: 12 000 and
# 40 000 for forces, 20 000 and 150 000 for energies; the FG reference (one
# list) and propane in its smallest box have the longest and shortest lists
SYSTEMS = {
    "propane_648": lambda: S.propane(),
    "fg_only_1250": lambda: S.fg_only(S.neopentane(n_mol=250, seed=6)),
    "neopentane_10000": lambda: S.neopentane(n_mol=2000, seed=7),
    "neopentane_10005": lambda: S.neopentane(n_mol=2001, density=0.5, seed=8),
    "neopentane_16670": lambda: S.neopentane(n_mol=3334, density=0.5, seed=9),
    "neopentane_33330": lambda: S.neopentane(n_mol=6666, seed=10),
}


@pytest.mark.parametrize("name", list(SYSTEMS))
def test_lanes_keep_the_bits_of_one_thread(torch, name):
    s = SYSTEMS[name]()
    out = []
    for config in (-1, 0):
        ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
        ctx.set_pair_config(config)
        p, v = _dev(torch, s.pos), _dev(torch, s.vel)
        ctx.build_neighbors(p, s.box)
        th = torch.zeros((6, R.RELRES_THERMO_COLS), dtype=torch.float64, device="cuda")
        ctx.step(60, s.dt, p, v, t_target=s.temperature, tau_fs=100.0, seed=3, thermo_every=10, d_thermo=th)
        torch.cuda.synchronize()
        lists = [ctx.get_list(w) for w in ((2, 3) if s.n_hybrid else (2,))]
        out.append((p.cpu().numpy(), v.cpu().numpy(), th.cpu().numpy(), ctx.stats()["n_prunes"], lists))
        ctx.close()
    (p0, v0, t0, n0, l0), (p1, v1, t1, n1, l1) = out
    assert np.array_equal(p0, p1) and np.array_equal(v0, v1)
    assert np.array_equal(t0, t1)
    assert n0 == n1 and n0 > 2
    for a, b in zip(l0, l1):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("acc", [R.RELRES_ACC_FP32, R.RELRES_ACC_COMPENSATED, R.RELRES_ACC_FP64])
@pytest.mark.parametrize("prune", [0.5, 0.0])
def test_energies_and_virial_do_not_depend_on_accumulation_or_pruning(torch, acc, prune):
    from oracle import core as O

    s = S.neopentane(n_mol=400, seed=12)
    ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
    ctx.set_force_accumulation(acc)
    ctx.set_prune(prune)
    p = _dev(torch, s.pos)
    ctx.build_neighbors(p, s.box)
    f = torch.empty_like(p)
    e, w = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.zeros(6, dtype=torch.float64, device="cuda")
    ctx.compute(p, f, e, w)
    torch.cuda.synchronize()
    ctx.close()
    _, e0, w0 = O.pair_forces(s.pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    e, w = e.cpu().numpy(), w.cpu().numpy()
    assert abs(e[0] + e[1] - e0) <= 1e-7 * abs(e0)
    # FP32 products of each pair, summed exactly: a few 2^-24 of the largest component
    assert np.abs(w - w0).max() <= 2e-6 * np.abs(w0[:3]).max()
    # the bits of the default accumulation and pruning
    ref = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
    ref.build_neighbors(p, s.box)
    e1, w1 = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.zeros(6, dtype=torch.float64, device="cuda")
    ref.compute(p, f, e1, w1)
    torch.cuda.synchronize()
    ref.close()
    assert np.array_equal(e, e1.cpu().numpy()) and np.array_equal(w, w1.cpu().numpy())


def test_overlapping_atoms_keep_their_energy(torch):
    """A pair whose energy and virial are past the range of the FP32 conversion
    to fixed point (2^20 kcal/mol)."""
    from oracle import core as O

    s = S.propane()
    pos = s.pos.copy()
    pos[3] = pos[0] + np.array([0.5, 0.6, 0.4])  # atoms of two molecules, 0.88 A apart
    ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    p = _dev(torch, pos)
    ctx.build_neighbors(p, s.box)
    f = torch.empty_like(p)
    e, w = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.zeros(6, dtype=torch.float64, device="cuda")
    ctx.compute(p, f, e, w)
    torch.cuda.synchronize()
    ctx.close()
    _, e0, w0 = O.pair_forces(pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    assert abs(e0) > 2.0 ** 20
    assert abs(float(e[3]) - e0) <= 1e-7 * abs(e0)
    assert np.abs(w.cpu().numpy() - w0).max() <= 1e-5 * np.abs(w0).max()


def test_fp64_batch_keeps_the_bits_of_each_replica_alone(torch):
    """FP64 replicas that alone take eight lanes per list or more and together four."""
    systems = [S.neopentane(n_mol=1000, seed=31), S.propane(n_mol=1000, box=53.0, seed=32),
               S.neopentane(n_mol=2000, seed=33), S.neopentane(n_mol=400, seed=34)]
    temps, seeds = [s.temperature for s in systems], [5, 6, 7, 8]

    def make():
        out = []
        for s in systems:
            ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP64), R.topology_for(s))
            p, v = _dev(torch, s.pos), _dev(torch, s.vel)
            ctx.build_neighbors(p, s.box)
            out.append((ctx, p, v))
        return out

    alone = make()
    for (c, p, v), t, sd in zip(alone, temps, seeds):
        assert c.stats()["pair_tpa"] == 8
        c.step(60, 1.0, p, v, t_target=t, tau_fs=100.0, seed=sd)
    both = make()
    batch = R.Batch([c for c, _, _ in both])
    batch.step(60, 1.0, [p for _, p, _ in both], [v for _, _, v in both], temps, 100.0, seeds)
    torch.cuda.synchronize()
    assert batch.n_shared() == 4 and sum(s.n_atoms + s.n_hybrid for s in systems) > 19456
    for (c1, p1, v1), (c2, p2, v2) in zip(alone, both):
        assert np.array_equal(p1.cpu().numpy(), p2.cpu().numpy())
        assert np.array_equal(v1.cpu().numpy(), v2.cpu().numpy())
    batch.close()
    for c, _, _ in alone + both:
        c.close()


def test_fp64_lanes_by_size_keep_the_bits(torch):
    """32, 32, 16 and 8 threads per slot alone (energy steps 32, 32, 16 and 16), four in one batch."""
    systems = [S.propane(), S.neopentane(n_mol=400, seed=41), S.neopentane(n_mol=1000, seed=42),
               S.neopentane(n_mol=2000, seed=43)]

    def run(batched):
        ctxs, ps, vs, ths = [], [], [], []
        for s in systems:
            ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP64), R.topology_for(s))
            ps.append(_dev(torch, s.pos))
            vs.append(_dev(torch, s.vel))
            ths.append(torch.zeros((6, R.RELRES_THERMO_COLS), dtype=torch.float64, device="cuda"))
            ctx.build_neighbors(ps[-1], s.box)
            ctxs.append(ctx)
        if batched:
            b = R.Batch(ctxs)
            b.step(30, 1.0, ps, vs, [0.0] * 4, 100.0, [1] * 4, thermo_every=5, d_thermo=ths)
            assert b.n_shared() == 4
            b.close()
        else:
            for c, p, v, th in zip(ctxs, ps, vs, ths):
                c.step(30, 1.0, p, v, thermo_every=5, d_thermo=th)
        torch.cuda.synchronize()
        for c in ctxs:
            c.close()
        return [[x.cpu().numpy() for x in (p, v, th)] for p, v, th in zip(ps, vs, ths)]

    for (p0, v0, t0), (p1, v1, t1) in zip(run(False), run(True)):
        assert np.array_equal(p0, p1) and np.array_equal(v0, v1)
        # pair energies summed in groups of 32 / T slots and rounded to 2^-52 kcal/mol per group or better
        assert np.abs(t0 - t1).max() <= 1e-12 * np.abs(t0).max()


# around the changes of the rules: threads per list of forces-only launches, of launches with energies, and the
# launch configuration that relres_stats names
@pytest.mark.parametrize("precision, n_mol, forces, energies, config", [
    (R.RELRES_PREC_FP64, 400, (32, 32), (32, 32), (8, 32)),       # 2 400 atoms and hybrids
    (R.RELRES_PREC_FP64, 1000, (16, 32), (16, 32), (8, 32)),      # 6 000
    (R.RELRES_PREC_FP64, 2000, (8, 32), (16, 32), (8, 32)),       # 12 000
    (R.RELRES_PREC_FP64, 3300, (4, 32), (4, 32), (4, 32)),        # 19 800
    (R.RELRES_PREC_FP32, 2000, (8, 128), (8, 128), (1, 256)),     # 12 000
    (R.RELRES_PREC_FP32, 2001, (4, 128), (8, 128), (1, 256)),
    (R.RELRES_PREC_FP32, 6666, (4, 128), (4, 128), (1, 256)),     # 39 996
])
def test_the_reported_launch_is_the_one_that_runs(torch, precision, n_mol, forces, energies, config):
    s = S.neopentane(n_mol=n_mol, density=0.5, seed=3)
    ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    with pytest.raises(R.RelresError) as ei:
        R.relres_get_pair_launch(ctx.ctx)
    assert ei.value.status == 6
    p = _dev(torch, s.pos)
    ctx.build_neighbors(p, s.box)
    f = torch.empty_like(p)
    for _ in range(2):  # before and after the first evaluation
        assert R.relres_get_pair_launch(ctx.ctx) == forces and R.relres_get_pair_launch(ctx.ctx, True) == energies
        st = ctx.stats()
        assert (st["pair_tpa"], st["pair_block"]) == config
        ctx.compute(p, f)
    if precision == R.RELRES_PREC_FP32:  # a fixed configuration, and accumulations that no lanes share
        ctx.set_pair_config(4)
        assert R.relres_get_pair_launch(ctx.ctx) == (4, 256) and R.relres_get_pair_launch(ctx.ctx, True) == energies
        ctx.set_pair_config(-1)
        ctx.set_force_accumulation(R.RELRES_ACC_FP64)
        assert R.relres_get_pair_launch(ctx.ctx)[0] == 1 and R.relres_get_pair_launch(ctx.ctx, True) == (1, 128)
    ctx.close()


def test_the_autotuner_times_launches_above_the_sizes_with_a_rule(torch):
    """42 000 atoms and hybrids: with pruning one thread per list, in blocks that the timing chose; 36 000 take four
    lanes without timing."""
    for n_mol, threads in ((6000, 4), (7000, 1)):
        s = S.neopentane(n_mol=n_mol, seed=2)
        ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
        p, v = _dev(torch, s.pos), _dev(torch, s.vel)
        ctx.build_neighbors(p, s.box)
        n0 = ctx.stats()["n_launches"]
        ctx.step(2, s.dt, p, v)
        st = ctx.stats()
        launch = R.relres_get_pair_launch(ctx.ctx)
        assert launch[0] == threads
        if threads == 1:
            # three configurations, four launches each
            assert launch == (1, st["pair_block"]) and launch[1] in (128, 256, 512)
            assert st["n_launches"] - n0 > 12
        ctx.close()


def with_copied_types(s, copies):
    """The same system with every type present `copies` times, atoms spread over the copies."""
    nt = s.n_types
    pick = np.random.default_rng(0).integers(0, copies, s.n_atoms)
    comp = np.zeros((nt * copies, nt * copies), np.int32)
    for q in range(copies):
        comp[q * nt:(q + 1) * nt, :nt] = np.asarray(s.group_comp).reshape(nt, nt)
    rep = lambda a: np.tile(np.asarray(a), copies)
    return s.subset_copy(types=(s.types + nt * pick).astype(np.int32), eps_fg=rep(s.eps_fg), sig_fg=rep(s.sig_fg),
                         is_hybrid=rep(s.is_hybrid).astype(np.int32), group_comp=comp,
                         mass_by_type=rep(s.mass_by_type))


# 32, 16, 8 and 4 threads per list; up to two types a launch of four copies the
# parameter rows to shared memory, else they are read in place
@pytest.mark.parametrize("n_mol", [130, 1000, 2000, 4000])
@pytest.mark.parametrize("copies", [2, 4])
def test_fp64_results_do_not_depend_on_where_the_parameters_are_read(torch, n_mol, copies):
    base = S.neopentane(n_mol=n_mol, density=0.5, seed=3)
    out = []
    for s in (base, with_copied_types(base, copies)):
        ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP64), R.topology_for(s))
        p = _dev(torch, s.pos)
        ctx.build_neighbors(p, s.box)
        f, g = torch.empty_like(p), torch.empty_like(p)
        e, w = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.zeros(6, dtype=torch.float64, device="cuda")
        ctx.compute(p, f)
        ctx.compute(p, g, e, w)
        p, v = _dev(torch, s.pos), _dev(torch, s.vel)
        batch = R.Batch([ctx])  # the same kernels with their arguments in device memory
        batch.set_mode(1)
        batch.step(5, 1.0, [p], [v], [0.0], 100.0, [1])
        torch.cuda.synchronize()
        batch.close()
        ctx.close()
        out.append([x.cpu().numpy() for x in (f, g, e, w, p, v)])
    assert np.array_equal(out[0][0], out[0][1])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
