"""FP64 contexts at the limits of the regions (r_s-, r_s+, r_c-, r_c+): pairs of
hybrid atoms 1e-8 A on either side of one, where an FP32 distance cannot tell
the side.  Without the full shift ("shift no") the CG energy jumps at r_c+ by
f_{c-}(r_c+ - r_c-); everything else is continuous."""
import numpy as np
import pytest

from oracle import core as O
from oracle import params as P
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


def _pairs_at(r, cells, seed):
    """A lattice whose sites are joined into pairs at r +- 1e-8 A: neighbours along x, or next neighbours (long r)."""
    rng = np.random.default_rng(seed)
    step = 2 if r > 10.0 else 1
    a = r / step
    k = np.stack(np.meshgrid(*[np.arange(c) for c in cells], indexing="ij"), -1).reshape(-1, 3)
    pos = a * (k + 0.5) + rng.uniform(-0.05, 0.05, k.shape) * a
    first = (k[:, 0] // step) % 2 == 0
    partner = {tuple(q): i for i, q in enumerate(k)}
    i = np.nonzero(first)[0]
    j = np.array([partner[(q[0] + step, q[1], q[2])] for q in k[i]])
    d = pos[j] - pos[i]
    d /= np.linalg.norm(d, axis=1)[:, None]
    side = np.where(rng.random(len(i)) < 0.5, -1e-8, 1e-8)
    pos[j] = pos[i] + d * (r + side)[:, None]
    return pos, a * np.array(cells, float)


# 32, 16 and 4 threads per list
@pytest.mark.parametrize("cells", [(8, 7, 6), (16, 14, 12), (32, 28, 26)])
@pytest.mark.parametrize("limit", [0, 1, 2, 3])
@pytest.mark.parametrize("shift", [False, True])
def test_fp64_regions_follow_the_fp64_distance(torch, cells, limit, shift):
    base = S.neopentane(n_mol=8)
    r = base.radii[limit]
    pos, box = _pairs_at(r, cells, seed=limit)
    n = len(pos)
    hyb = int(np.nonzero(base.is_hybrid)[0][0])
    types = np.full(n, hyb, np.int32)
    tab = P.pair_table(base.eps_fg, base.sig_fg, base.is_hybrid, base.radii, mixing=base.mixing,
                       group_comp=base.group_comp, shift=shift)
    off, idx = np.zeros(n + 1, np.int32), np.zeros(0, np.int32)
    fr, e0, w0 = O.pair_forces(pos, box, types, tab, base.n_types, (off, idx))
    ctx = R.Context(R.params_for(base, R.RELRES_PREC_FP64, shift=shift),
                    R.make_topology(types, base.mass_by_type, (off, idx), None))
    x = torch.tensor(pos, dtype=torch.float64, device="cuda")
    ctx.build_neighbors(x, box)
    f, g = torch.empty_like(x), torch.empty_like(x)
    e = torch.zeros(4, dtype=torch.float64, device="cuda")
    w = torch.zeros(6, dtype=torch.float64, device="cuda")
    for _ in range(2):  # as the pair launch prunes, and on the pruned lists
        ctx.compute(x, f, e, w)
        torch.cuda.synchronize()
        assert abs(float(e[3]) - e0) <= 1e-12 * abs(e0), (float(e[3]), e0)
        assert np.abs(f.cpu().numpy() - fr).max() <= 1e-10 * np.sqrt((fr * fr).sum(1).mean())
        assert np.abs(w.cpu().numpy() - w0).max() <= 1e-11 * np.abs(w0).max()
    ctx.compute(x, g)
    torch.cuda.synchronize()
    assert np.array_equal(f.cpu().numpy(), g.cpu().numpy())
    ctx.close()
    if limit == 3 and not shift:
        # the jump, so that the case does tell the sides apart
        t = tab[hyb * base.n_types + hyb]
        ws = base.radii[3] - base.radii[2]
        jump = abs((((t[22] * ws + t[21]) * ws + t[20]) * ws + t[19]) * ws + t[18])
        assert jump > 1e-3 and jump > 1e-9 * abs(e0)
