"""Coincident points without a nugget make a unit's matrix exactly singular.  Every kernel that factors units reports
SIC_ERR_NOT_PD for any such pair, at a variance that is no power of two, whichever launch the number or the size
of the units selects; with a nugget the same units have a factor."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401
from test_gpu_unit_precision import _partial

pytestmark = pytest.mark.gpu
N = 24


def _cases(k):
    """Pairs (i, j) of one unit's N points that are made to coincide."""
    r = np.random.RandomState(5)
    return [tuple(sorted(r.choice(N, 2, replace=False))) for _ in range(k)]


def _status(sic, f):
    try:
        f()
    except sic.SicError as e:
        return e.code
    return 0


@pytest.mark.parametrize("nugget", [0.0, 1e-4])
def test_partial_fill(env, nugget):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.3, 1.3, nugget)
    want = 0 if nugget else sic.SIC_ERR_NOT_PD
    for i, j in _cases(30):
        pts = synthetic.points(N, 2, 21)
        pts[j] = pts[i]
        assert _status(sic, lambda: _partial(env, pts, kp, [(np.arange(0, N, 2), np.arange(1, N, 2))], 12)) == want


@pytest.mark.parametrize("nugget", [0.0, 1e-4])
@pytest.mark.parametrize("units", [3, 1800])  # the flat kernel and the panels
def test_side_state(env, nugget, units):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.3, 1.3, nugget)
    want = 0 if nugget else sic.SIC_ERR_NOT_PD
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    sel = d(np.tile(np.arange(1, N, dtype=np.int32), units))
    out = torch.zeros(units * (N - 1), dtype=torch.float64, device="cuda")
    for i, j in _cases(12):
        pts = synthetic.points(N, 2, 21)
        pts[j] = pts[i]

        def call():
            sic.side_state_fp64(h, d(pts), kp, sel, d(np.full(units, N - 1, np.int32)), N - 1,
                                targets=d(np.zeros(units, np.int32)), gain=out)
            h.sync()
        assert _status(sic, call) == want


@pytest.mark.parametrize("nugget", [0.0, 1e-4])
@pytest.mark.parametrize("grouped,k", [(False, 20), (False, 49), (True, 20)])
def test_fill(env, nugget, grouped, k):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.3, 1.3, nugget)
    want = 0 if nugget else sic.SIC_ERR_NOT_PD
    for i, j in _cases(12):
        pts = synthetic.points(N, 2, 21)
        pts[j] = pts[i]
        m = 4 if grouped else 1
        gp = np.concatenate([np.arange(0, N, m), [N]]).astype(np.int64)
        ptr = np.zeros(len(gp), np.int64)
        hp = pipeline.HostProblem(pts, kp, k, ptr, np.zeros(0, np.int32), gp if grouped else None)
        b = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
        sel = np.full((hp.n_units, k), -1, np.int32)
        cnt = np.array([min(k, N - int(gp[u + 1])) for u in range(hp.n_units)], np.int32)
        for u in range(hp.n_units):  # every later point
            sel[u, :cnt[u]] = np.arange(gp[u + 1], gp[u + 1] + cnt[u])
        if not grouped and j > i + k:
            continue  # the pair shares no column
        b.sel_idx.copy_(torch.from_numpy(sel.reshape(-1)))
        b.sel_count.copy_(torch.from_numpy(cnt))

        def call():
            b.fill(pipeline.DeviceProblem(hp))
            h.sync()
        assert _status(sic, call) == want
