"""Force evaluations as calls of their own (relres_compute, relres_backward):
lists refreshed on the device without a host round trip.  Positions past the
rebuild trigger, lists that overflow inside the evaluation, pruning left over
by a build, and non-finite positions, which leave the outputs alone."""
import numpy as np
import pytest

from oracle import core as O
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


def _reference(s, pos):
    fr, e, _ = O.pair_forces(pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    fb, _ = O.bonded(pos, s.box, s.topo)
    return fr + fb, e


def _err(f, ref):
    return np.abs(f - ref).max() / np.sqrt((ref * ref).sum(1).mean())


# a shift of every atom by more than half the skin rebuilds without changing
# the physics; 25 000 atoms take the launches chosen by timing
@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
@pytest.mark.parametrize("n_mol", [250, 1000])
@pytest.mark.parametrize("config", [-1, 3])
def test_moved_positions_rebuild_inside_the_evaluation(torch, precision, n_mol, config):
    s = S.neopentane(n_mol=n_mol, seed=4)
    ctx = R.Context(R.params_for(s, precision), R.topology_for(s))
    ctx.set_pair_config(config)
    ctx.build_neighbors(_dev(torch, s.pos), s.box)
    ref, e0 = _reference(s, s.pos)
    tol = 1e-5 if precision == R.RELRES_PREC_FP32 else 1e-10
    builds = ctx.stats()["n_builds"]
    for k, shift in enumerate((0.0, 0.4, 1.5, 1.6, 7.0)):
        x = _dev(torch, s.pos + shift)
        f, e = torch.empty_like(x), torch.zeros(4, dtype=torch.float64, device="cuda")
        ctx.compute(x, f, e)
        torch.cuda.synchronize()
        assert _err(f.cpu().numpy(), ref) <= tol, shift
        assert abs(float(e[0] + e[1]) - e0) <= 1e-7 * abs(e0)
    st = ctx.stats()
    assert st["n_builds"] == builds + 2  # at 1.5 (from 0) and 7.0 (from 1.5)
    assert st["n_prunes"] >= st["n_builds"]
    ctx.close()


def test_overflow_inside_an_evaluation_grows_the_lists(torch):
    s = S.neopentane(n_mol=300, seed=5)
    ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
    ctx.build_neighbors(_dev(torch, s.pos * 1.0), s.box)
    f = _dev(torch, s.pos)
    ctx.compute(_dev(torch, s.pos), f)
    ctx.set_list_caps(1, 1)  # grown at once to what these positions need
    # half of the liquid pushed into half of the box: far longer lists
    pos = s.pos.copy()
    mol = s.mol
    centre = np.stack([s.pos[mol == m].mean(0) for m in range(mol.max() + 1)])
    pos += (np.floor(centre / s.box * 2) / 2 * -1)[mol] * s.box * np.array([0.0, 0.0, 0.97])
    x = _dev(torch, pos)
    e = torch.zeros(4, dtype=torch.float64, device="cuda")
    ctx.compute(x, f, e)
    torch.cuda.synchronize()
    ref, _ = _reference(s, np.mod(pos, s.box))
    assert _err(f.cpu().numpy(), ref) <= 1e-5
    ctx.close()


def test_nonfinite_positions_leave_outputs_and_lists_alone(torch):
    s = S.neopentane(n_mol=300, seed=6)
    ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP32), R.topology_for(s))
    good = _dev(torch, s.pos)
    ctx.build_neighbors(good, s.box)
    f = torch.empty_like(good)
    ctx.compute(good, f)
    want = f.cpu().numpy()
    bad = good.clone()
    bad[7, 1] = float("nan")
    e = torch.full((4,), 3.0, dtype=torch.float64, device="cuda")
    f.fill_(5.0)
    g = torch.full_like(good, 9.0)
    for call in (lambda: ctx.compute(bad, f, e), lambda: ctx.backward(bad, None, 1.0, g)):
        with pytest.raises(R.RelresError) as ei:
            call()
        assert ei.value.status == 5 and "position" in str(ei.value)
    torch.cuda.synchronize()
    assert float(f.min()) == float(f.max()) == 5.0 and float(e.min()) == 3.0 and float(g.min()) == 9.0
    ctx.compute(good, f)
    torch.cuda.synchronize()
    assert np.abs(f.cpu().numpy() - want).max() <= 1e-5 * np.abs(want).max()
    assert ctx.stats()["n_builds"] == 1
    ctx.close()


# A build leaves the pruning pass to the next evaluation; a non-finite position
# ends that evaluation before it, and the one after it prunes.  Configuration 3
# has the pass run by the rebuild kernel instead of the pair launch; 40 008
# atoms and hybrids is above the sizes whose launch shape goes without timing.
@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
@pytest.mark.parametrize("first", ["backward", "compute", "config", "tuned"])
def test_nonfinite_positions_right_after_a_build(torch, precision, first):
    s = S.neopentane(n_mol=6668 if first == "tuned" else 400, seed=8)
    ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    good = _dev(torch, s.pos)
    bad = good.clone()
    bad[s.n_atoms // 2, 2] = float("inf")
    ctx.build_neighbors(good, s.box)
    if first == "config":
        ctx.set_pair_config(3)
    f, g = torch.full_like(good, 5.0), torch.full_like(good, 9.0)
    e = torch.full((4,), 3.0, dtype=torch.float64, device="cuda")
    with pytest.raises(R.RelresError) as ei:
        if first == "backward":
            ctx.backward(bad, None, 1.0, g)
        else:
            ctx.compute(bad, f, e if first == "compute" else None)
    assert ei.value.status == 5 and "position" in str(ei.value)
    torch.cuda.synchronize()
    assert float(f.min()) == float(f.max()) == 5.0 and float(e.max()) == 3.0 and float(g.max()) == 9.0
    # a little further on, within the margin of both lists
    x = good + 0.2
    if first == "backward":
        ctx.backward(x, None, 1.0, g)
        f = -g
    else:
        ctx.compute(x, f, e)
    torch.cuda.synchronize()
    ref, e0, _ = O.pair_forces(s.pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    assert _err(f.cpu().numpy(), ref) <= (1e-5 if precision == R.RELRES_PREC_FP32 else 1e-10)
    if first != "backward":
        assert abs(float(e[3]) - e0) <= 1e-7 * abs(e0)
    assert ctx.stats()["n_builds"] == 1
    lists = [set(map(tuple, ctx.get_list(w).tolist())) for w in range(4)]
    # (no hybrid pairs between the two radii in some of these lattices)
    assert lists[2] and lists[2] < lists[0] and lists[3] and lists[3] <= lists[1]
    ctx.close()


@pytest.mark.parametrize("n_mol", [300, 1200])
def test_new_topology_after_a_build_and_before_an_evaluation(torch, n_mol):
    """The pruning pass left over by the first build goes with its lists."""
    s0, s = S.neopentane(n_mol=600, seed=9), S.neopentane(n_mol=n_mol, seed=10)
    ctx = R.Context(R.params_for(s0, R.RELRES_PREC_FP32), R.topology_for(s0))
    ctx.build_neighbors(_dev(torch, s0.pos), s0.box)
    ctx.set_topology(R.topology_for(s))
    assert ctx.stats()["n_prunes"] == 0
    for call in (lambda: ctx.get_list(2), lambda: ctx.compute(_dev(torch, s.pos), _dev(torch, s.pos))):
        with pytest.raises(R.RelresError) as ei:
            call()
        assert ei.value.status == 6
    x = _dev(torch, s.pos)
    ctx.build_neighbors(x, s.box)
    f, e = torch.empty_like(x), torch.zeros(4, dtype=torch.float64, device="cuda")
    ctx.compute(x, f, e)
    torch.cuda.synchronize()
    ref, e0 = _reference(s, s.pos)
    assert _err(f.cpu().numpy(), ref) <= 1e-5 and abs(float(e[0] + e[1]) - e0) <= 1e-7 * abs(e0)
    st = ctx.stats()
    assert st["n_prunes"] == 1 and st["n_atoms"] == s.n_atoms
    ctx.close()


def test_backward_right_after_a_build_reads_pruned_lists(torch):
    s = S.propane()
    ctx = R.Context(R.params_for(s, R.RELRES_PREC_FP64), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    x = _dev(torch, s.pos)
    ctx.build_neighbors(x, s.box)
    g = torch.empty_like(x)
    ctx.backward(x, None, 1.0, g)
    torch.cuda.synchronize()
    fr, _, _ = O.pair_forces(s.pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    assert _err(g.cpu().numpy(), -fr) <= 1e-10
    ctx.close()


def test_batch_calls_continue_or_read_the_arrays_as_each_replica_alone(torch):
    """Second and third calls with one replica's positions changed, another's velocities, another left alone, an
    FP64 one, then all with another time step: the bits of every context stepped by itself."""
    systems = [S.neopentane(n_mol=200, seed=51), S.propane(), S.neopentane(n_mol=120, seed=52), S.propane(seed=53)]
    prec = [R.RELRES_PREC_FP32] * 3 + [R.RELRES_PREC_FP64]

    def run(batched):
        ctxs, ps, vs = [], [], []
        for s, q in zip(systems, prec):
            ctxs.append(R.Context(R.params_for(s, q), R.topology_for(s)))
            ps.append(_dev(torch, s.pos))
            vs.append(_dev(torch, s.vel))
            ctxs[-1].build_neighbors(ps[-1], s.box)
        temps, seeds = [s.temperature for s in systems], [3, 4, 5, 6]
        batch = R.Batch(ctxs) if batched else None
        for call, dt in enumerate((1.0, 1.0, 0.5)):
            if call == 1:
                ps[0] += 0.01
                vs[1] *= 0.9
                vs[3] *= 1.1
            if batched:
                batch.step(7, dt, ps, vs, temps, 100.0, seeds)
            else:
                for c, p, v, t, sd in zip(ctxs, ps, vs, temps, seeds):
                    c.step(7, dt, p, v, t_target=t, tau_fs=100.0, seed=sd)
        torch.cuda.synchronize()
        if batched:
            batch.close()
        for c in ctxs:
            c.close()
        return [x.cpu().numpy() for x in ps + vs]

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)
