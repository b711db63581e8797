"""relres_pair_forces_static at the sizes where its warp-per-atom kernel can go
wrong (one atom, partial warps and blocks, partial queues), with positions in
other periodic images, without exclusions, with unequal box edges and with a
non-finite coordinate, against the FP64 oracle's all-pairs sum of Eq. 20."""
import math

import numpy as np
import pytest

from paper_2104_10231_gb300 import relres as R
from paper_2104_10231_gb300 import systems as S

pytestmark = pytest.mark.gpu

# FP64 sums of up to a few thousand terms in another order: n_terms * 2^-53
# relative to the largest partial sums, with room for close pairs
TOL = 1e-11


@pytest.fixture(scope="module")
def torch():
    import torch as T

    assert T.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2104_10231_gb300.build import build_library

    build_library()
    R.load()
    return T


def _atoms(n, box, n_types, seed):
    """n atoms at least 3 A apart in the box, some displaced by whole box edges."""
    rng = np.random.default_rng(seed)
    pos = np.zeros((0, 3))
    while len(pos) < n:
        x = rng.random((1, 3)) * box
        d = pos - x
        d -= box * np.round(d / box)
        if len(pos) == 0 or (d * d).sum(1).min() > 9.0:
            pos = np.concatenate([pos, x])
    types = rng.integers(0, n_types, n).astype(np.int32)
    return pos + box * rng.integers(-3, 4, (n, 3)), types


def _call(torch, params, pos, types, box, excl, energy=True):
    dev = lambda a, dt: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    f = torch.full((len(pos), 3), 7.0, dtype=torch.float64, device="cuda")
    e = torch.full((1,), 7.0, dtype=torch.float64, device="cuda")
    w = torch.full((6,), 7.0, dtype=torch.float64, device="cuda")
    ex = (None, None) if excl is None else (dev(excl[0], torch.int32), dev(excl[1], torch.int32))
    R.relres_pair_forces_static(params, len(pos), dev(types, torch.int32), dev(pos, torch.float64), box, f,
                                e if energy else None, w if energy else None, *ex)
    torch.cuda.synchronize()
    return f.cpu().numpy(), float(e[0]), w.cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 5, 31, 32, 33, 127, 130, 260, 1029])
@pytest.mark.parametrize("with_excl", [False, True])
def test_static_at_partial_warps_blocks_and_queues(torch, n, with_excl):
    from oracle import core as O

    s = S.propane()
    box = np.array([29.0, 36.0, 47.0]) if n < 500 else np.array([40.0, 36.0, 47.0])
    pos, types = _atoms(n, box, s.n_types, n)
    excl = (np.zeros(n + 1, np.int32), np.zeros(0, np.int32))
    if with_excl:  # consecutive atoms in runs of three, as in the liquid
        mol = np.arange(n) // 3
        part = [[j for j in range(max(0, i - 2), min(n, i + 3)) if j != i and mol[j] == mol[i]] for i in range(n)]
        excl = (np.cumsum([0] + [len(p) for p in part]).astype(np.int32),
                np.array([j for p in part for j in p], np.int32))
    f0, e0, w0 = O.pair_forces(pos, box, types, O.table_for(s), s.n_types, excl)
    params = R.params_for(s, R.RELRES_PREC_FP64)
    f, e, w = _call(torch, params, pos, types, box, excl if len(excl[1]) else None)
    scale = max(1e-3, float(np.abs(f0).max()))
    assert np.abs(f - f0).max() <= TOL * scale
    assert abs(e - e0) <= TOL * max(1.0, abs(e0))
    assert np.abs(w - w0).max() <= TOL * max(1.0, float(np.abs(w0).max()))
    f2, e2, w2 = _call(torch, params, pos, types, box, excl if len(excl[1]) else None, energy=False)
    assert np.array_equal(f2, f) and e2 == 7.0 and (w2 == 7.0).all()  # outputs not asked for stay untouched


def test_static_passes_a_nonfinite_coordinate_on(torch):
    s = S.propane()
    box = np.array([40.0, 36.0, 47.0])
    pos, types = _atoms(100, box, s.n_types, 3)
    pos[41, 1] = math.inf
    f, _, w = _call(torch, R.params_for(s, R.RELRES_PREC_FP64), pos, types, box, None)
    assert np.isnan(f).any(axis=1).all() and np.isnan(w).any()
