"""FP64 angle terms where their evaluation changes over: theta - theta0 from the
arcsine series up to |sin(theta - theta0)| = 1/4 and from both components
beyond, and angles close to straight or closed, where the force goes as
1 / sin(theta).  Reference: the same term in extended precision."""
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


def _reference(pos, k, theta0):
    """Forces and energy of one angle per row of pos (n, 3 atoms, 3); also sin(theta)."""
    p = pos.astype(np.longdouble)
    r1, r2 = p[:, 0] - p[:, 1], p[:, 2] - p[:, 1]
    n1, n2 = (np.sqrt((r * r).sum(1)) for r in (r1, r2))
    u1, u2 = r1 / n1[:, None], r2 / n2[:, None]
    s = np.sqrt((np.cross(u1, u2) ** 2).sum(1))
    c = (u1 * u2).sum(1)
    d = np.arctan2(s, c) - theta0
    q1, q2 = (u2 - c[:, None] * u1) / s[:, None], (u1 - c[:, None] * u2) / s[:, None]  # towards the other arm
    f0, f2 = (2 * k * d / n1)[:, None] * q1, (2 * k * d / n2)[:, None] * q2
    return np.stack([f0, -(f0 + f2), f2], 1).astype(float), float((k * d * d).sum()), s.astype(float)


def _angles(theta0):
    a = np.arcsin(0.25)
    t = [theta0 + sign * (a + e) for sign in (1, -1) for e in (0.0, 1e-15, -1e-15, 1e-9, -1e-9, 1e-3, -1e-3)]
    t += [theta0, theta0 + 1e-9, theta0 - 1e-6, theta0 + np.pi / 2, theta0 - np.pi / 2, theta0 + 3.0, theta0 - 3.0]
    t += [np.pi - e for e in (1e-4, 1e-3, 0.1)] + [1e-4, 1e-3, 0.1]
    t = np.array(t)
    return t[(t > 5e-5) & (t < np.pi - 5e-5)]


@pytest.mark.parametrize("segments", [True, False])
@pytest.mark.parametrize("degrees", [20.0, 90.0, 109.5, 165.0, 179.0])
def test_fp64_angles_at_the_changeovers(torch, degrees, segments):
    theta0, k = np.deg2rad(degrees), 60.0
    theta = np.tile(_angles(theta0), 6)
    m = len(theta)
    rng = np.random.default_rng(5)
    # one molecule of three atoms per angle, 12 A apart (past r_s+ of the FG sites)
    side = int(np.ceil(m ** (1 / 3)))
    grid = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:m]
    u = rng.normal(size=(m, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    w = np.cross(u, rng.normal(size=(m, 3)))
    w /= np.linalg.norm(w, axis=1)[:, None]
    centre = 12.0 * grid + 6.0
    arm = rng.uniform(1.3, 1.7, (m, 2, 1))
    pos = np.stack([centre + arm[:, 0] * u, centre,
                    centre + arm[:, 1] * (np.cos(theta)[:, None] * u + np.sin(theta)[:, None] * w)], 1)
    base = S.neopentane(n_mol=8)
    n = 3 * m
    bead = int(np.nonzero(np.asarray(base.is_hybrid) == 0)[0][0])
    i0 = 3 * np.arange(m)
    excl = np.stack([i0 + 1, i0 + 2, i0, i0 + 2, i0, i0 + 1], 1).reshape(-1).astype(np.int32)
    off = (2 * np.arange(n + 1)).astype(np.int32)
    topo = dict(bonds=np.zeros((0, 2), np.int32), bond_type=np.zeros(0, np.int32), bond_k=np.zeros(0), bond_r0=np.zeros(0),
                angles=np.stack([i0, i0 + 1, i0 + 2], 1).astype(np.int32), angle_type=np.zeros(m, np.int32),
                angle_k=np.array([k]), angle_theta0=np.array([theta0]), dihedrals=np.zeros((0, 4), np.int32),
                dihedral_type=np.zeros(0, np.int32), dihedral_k=np.zeros((0, 4)))
    box = np.full(3, max(12.0 * side, 36.0))
    order = np.arange(n)
    if not segments:
        # the ends of each angle 2 m atoms apart: whole molecules only in runs longer than a segment
        order = order.reshape(m, 3).T.reshape(-1)
        new = np.empty(n, np.int64)
        new[order] = np.arange(n)
        topo["angles"] = new[topo["angles"]].astype(np.int32)
        excl = np.concatenate([np.sort(new[excl[off[o]:off[o + 1]]]) for o in order]).astype(np.int32)
    ctx = R.Context(R.params_for(base, R.RELRES_PREC_FP64),
                    R.make_topology(np.full(n, bead, np.int32), base.mass_by_type, (off, excl), topo))
    flat = pos.reshape(n, 3)[order]
    x = torch.tensor(flat, dtype=torch.float64, device="cuda")
    ctx.build_neighbors(x, box)
    assert bool(ctx.stats()["step_segments"]) == segments
    f, e = torch.empty_like(x), torch.zeros(4, dtype=torch.float64, device="cuda")
    ctx.compute(x, f, e)
    torch.cuda.synchronize()
    ctx.close()
    got = np.empty((n, 3))
    got[order] = f.cpu().numpy()
    ref, e0, s = _reference(pos, k, theta0)
    assert float(e[0]) == 0.0 and abs(float(e[2]) - e0) <= 1e-10 * e0
    # coordinates of up to 100 A carry 2^-46 A; over the arms (1.3 A) and sin(theta) that is the direction's error,
    # and theta itself is off by it too
    eps = 100.0 * 2.0 ** -46 / 1.3
    scale = 2.0 * k * np.abs(theta - theta0) / 1.3
    tol = 8.0 * eps * (scale / s + 2.0 * k) + 1e-12
    assert (np.abs(got.reshape(m, 3, 3) - ref).max((1, 2)) <= tol).all(), np.abs(got.reshape(m, 3, 3) - ref).max((1, 2)) / tol
