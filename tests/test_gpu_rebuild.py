"""The list rebuild inside one kernel (its phases separated by a grid-wide
barrier with a bounded wait): rebuilds, pruning and overflows that come with a
backward pass, and the error path when the wait runs out."""
import time

import numpy as np
import pytest

from oracle import core as O
from paper_2104_10231_gb300 import relres as R
from paper_2104_10231_gb300 import systems as S
from tests.test_gpu_lanes import with_copied_types

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


def _pair_reference(s, pos):
    fr, e, _ = O.pair_forces(pos, s.box, s.types, O.table_for(s), s.n_types, s.excl)
    return fr, e


def _err(f, ref):
    return np.abs(f - ref).max() / np.sqrt((ref * ref).sum(1).mean())


def _backward(torch, ctx, s, pos):
    """Gradients of E for the box and lists of ctx at pos: dL/dx = -F, and the parameter gradients."""
    x = _dev(torch, pos)
    g = torch.empty_like(x)
    out = ctx.backward(x, None, 1.0, g)
    torch.cuda.synchronize()
    return g.cpu().numpy(), out


# shifts of the whole liquid leave the physics alone; the second and the last
# are past half the skin
@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
@pytest.mark.parametrize("n_mol", [250, 2334, 8334])  # 8, 4 and 2 threads per list in FP32
def test_backward_rebuilds_and_prunes_at_moved_positions(torch, precision, n_mol):
    s = S.neopentane(n_mol=n_mol, seed=12)
    ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    ctx.build_neighbors(_dev(torch, s.pos), s.box)
    ref, _ = _pair_reference(s, s.pos)
    first = None
    for shift in (0.0, 1.5, 1.7, 9.0):
        g, out = _backward(torch, ctx, s, s.pos + shift)
        assert _err(g, -ref) <= (1e-5 if precision == R.RELRES_PREC_FP32 else 1e-10), shift
        first = first or out
        # sums over all pairs of terms rounded to FP32 (FP64) once each
        tol = 1e-5 if precision == R.RELRES_PREC_FP32 else 1e-11
        for k, v in first.items():
            assert np.abs(out[k] - v).max() <= tol * np.abs(v).max(), (shift, k)
    st = ctx.stats()
    assert st["n_builds"] == 3 and st["n_prunes"] >= 3
    # the pruned lists of the rebuild kernel are those of a new context at the same positions
    got = [set(map(tuple, ctx.get_list(w).tolist())) for w in (2, 3)]
    ctx.close()
    new = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    new.build_neighbors(_dev(torch, s.pos + 9.0), s.box)
    want = [set(map(tuple, new.get_list(w).tolist())) for w in (2, 3)]
    new.close()
    assert got == want


@pytest.mark.parametrize("n_mol, copies", [(40000, 1), (14000, 4)])
def test_backward_of_a_large_system_with_one_thread_per_list(torch, n_mol, copies):
    """240 000 atoms and hybrids of two types and 84 000 of eight, FP32 against FP64 (two threads per list)."""
    s = with_copied_types(S.neopentane(n_mol=n_mol, density=0.5, seed=12), copies)
    rng = np.random.default_rng(1)
    gf = _dev(torch, rng.normal(size=s.pos.shape))
    out = []
    for precision in (R.RELRES_PREC_FP32, R.RELRES_PREC_FP64):
        ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
        x = _dev(torch, s.pos)
        ctx.build_neighbors(x, s.box)
        g = torch.empty_like(x)
        res = ctx.backward(x, gf, 1.0, g)
        torch.cuda.synchronize()
        out.append((g.cpu().numpy(), res))
        ctx.close()
    (g0, r0), (g1, r1) = out
    assert _err(g0, g1) <= 1e-5
    for k in r1:
        assert np.abs(r0[k] - r1[k]).max() <= 1e-5 * np.abs(r1[k]).max(), k


@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
def test_backward_grows_lists_that_overflow(torch, precision):
    s = S.neopentane(n_mol=300, seed=5)
    ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    ctx.build_neighbors(_dev(torch, s.pos), s.box)
    ctx.set_list_caps(1, 1)  # grown at once to what these positions need
    caps = ctx.stats()
    # half of the liquid pushed into half of the box: far longer lists
    centre = np.stack([s.pos[s.mol == m].mean(0) for m in range(s.mol.max() + 1)])
    pos = s.pos - np.floor(centre / s.box * 2)[s.mol] / 2 * s.box * np.array([0.0, 0.0, 0.97])
    g, _ = _backward(torch, ctx, s, pos)
    ref, _ = _pair_reference(s, np.mod(pos, s.box))
    assert _err(g, -ref) <= (1e-5 if precision == R.RELRES_PREC_FP32 else 1e-10)
    st = ctx.stats()
    assert st["cap_fg"] > caps["cap_fg"] and st["cap_cg"] > caps["cap_cg"]
    ctx.close()


def _stall(ctx):
    R._check(R.load().relres_stall_rebuild(ctx.ctx), ctx.ctx)


def _whole_again(torch, ctx, s, precision):
    """After the error the lists have to be built again; then everything is as in a new context."""
    x = _dev(torch, s.pos)
    f, e = torch.empty_like(x), torch.zeros(4, dtype=torch.float64, device="cuda")
    with pytest.raises(R.RelresError) as ei:
        ctx.compute(x, f, e)
    assert ei.value.status == 6
    ctx.stats()
    ctx.build_neighbors(x, s.box)
    ref, e0 = _pair_reference(s, s.pos)
    for shift in (0.0, 1.5, 0.0):  # the second and third rebuild inside the call
        ctx.compute(_dev(torch, s.pos + shift), f, e)
        torch.cuda.synchronize()
        assert _err(f.cpu().numpy(), ref) <= (1e-5 if precision == R.RELRES_PREC_FP32 else 1e-10)
        assert abs(float(e[3]) - e0) <= 1e-7 * abs(e0)


@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
@pytest.mark.parametrize("call", ["compute", "backward", "config"])
def test_barrier_that_runs_out_of_time_in_an_evaluation(torch, precision, call):
    s = S.neopentane(n_mol=500, seed=14)
    ctx = R.Context(R.params_for(s, precision), R.make_topology(s.types, s.mass_by_type, s.excl, None))
    if call == "config":
        ctx.set_pair_config(3)
    x = _dev(torch, s.pos)
    ctx.build_neighbors(x, s.box)
    _stall(ctx)
    out = torch.full_like(x, 5.0)
    e = torch.full((4,), 3.0, dtype=torch.float64, device="cuda")
    moved = x + 1.5  # past half the skin
    t0 = time.perf_counter()
    with pytest.raises(R.RelresError) as ei:
        if call == "backward":
            ctx.backward(moved, None, 1.0, out)
        else:
            ctx.compute(moved, out, e)
    assert time.perf_counter() - t0 < 20.0
    assert ei.value.status == 2 and "barrier" in str(ei.value)
    torch.cuda.synchronize()
    assert float(out.min()) == float(out.max()) == 5.0 and float(e.min()) == float(e.max()) == 3.0
    _whole_again(torch, ctx, s, precision)
    ctx.close()


@pytest.mark.parametrize("precision", [R.RELRES_PREC_FP32, R.RELRES_PREC_FP64])
def test_barrier_that_runs_out_of_time_in_a_step_returns_the_block_start(torch, precision):
    """The first rebuild of a run comes within its first block of 100 steps; the call gives back the arrays that it
    was given, through 64-bit fixed point (2^-64 of the box) and, in FP32 mode, float-float (2^-47)."""
    s = S.neopentane(n_mol=500, seed=31)
    ctx = R.Context(R.params_for(s, precision), R.topology_for(s))
    p, v = _dev(torch, np.mod(s.pos, s.box)), _dev(torch, s.vel)
    ctx.build_neighbors(p, s.box)
    ctx.step(1, 2.0, p, v, t_target=260.0, tau_fs=100.0, seed=4)
    p0, v0 = p.cpu().numpy(), v.cpu().numpy()
    _stall(ctx)
    with pytest.raises(R.RelresError) as ei:
        ctx.step(100, 2.0, p, v, t_target=260.0, tau_fs=100.0, seed=4)
    assert ei.value.status == 2 and "barrier" in str(ei.value)
    torch.cuda.synchronize()
    assert np.abs(p.cpu().numpy() - p0).max() <= 1e-12 * s.box.max()
    assert np.abs(v.cpu().numpy() - v0).max() <= 1e-13 * np.abs(v0).max()
    # on from there as a new context goes from the same arrays
    p2, v2 = _dev(torch, p.cpu().numpy()), _dev(torch, v.cpu().numpy())
    new = R.Context(R.params_for(s, precision), R.topology_for(s))
    for c, q, w in ((ctx, p, v), (new, p2, v2)):
        c.build_neighbors(q, s.box)
        R.relres_set_step_counter(c.ctx, 1)
        c.step(100, 2.0, q, w, t_target=260.0, tau_fs=100.0, seed=4)
    torch.cuda.synchronize()
    assert np.array_equal(p.cpu().numpy(), p2.cpu().numpy()) and np.array_equal(v.cpu().numpy(), v2.cpu().numpy())
    ctx.close()
    new.close()
