"""Precision of the units that are factored in FP64 throughout: the fill of nonadjacent groups and the FP64 side state,
against NumPy's long double (128 bits where these tests run).

Tolerances.  u = 2^-53.  Moderately correlated points (length scale a third of the mean distance, nugget 1e-2): Theta's
entries carry 2 ulp, the diagonal entry of a column, its largest, one reciprocal root of them and its rounding, so 6 u
on average over the columns covers both with every substitution step in FP64; factors held to 48 bits are off by
2^-48 = 32 u of their entries.  A point far
out has no covariance with the others, so it changes no bit of the pivots before its own; where it comes first in
the order the columns keep the error of the same unit without it, at nugget 1e-2 below 1e-12 (fewer than 100
steps of 1 / nugget u each), while coordinates cut 2^-61 below 2^34 would put them off by 1e-8."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu
LD = np.longdouble
FAR = float(2 ** 34)


def _theta(kp, X):
    X = X.astype(LD)
    r = np.sqrt(sum((X[:, None, d] - X[None, :, d]) ** 2 for d in range(X.shape[1])))
    t = np.sqrt(LD(kp.nu_x2)) * r / LD(kp.length_scale)
    p = {1: 1 + 0 * t, 3: 1 + t, 5: 1 + t + t * t / 3}[kp.nu_x2]
    return LD(kp.variance) * p * np.exp(-t) + LD(kp.nugget) * np.eye(len(X), dtype=LD)


def _ldl(A):
    A = A.copy()
    n = len(A)
    L = np.eye(n, dtype=LD)
    d = np.zeros(n, dtype=LD)
    for j in range(n):
        d[j] = A[j, j]
        L[j + 1:, j] = A[j + 1:, j] / d[j]
        A[j + 1:, j + 1:] -= np.outer(L[j + 1:, j], A[j, j + 1:])
        A[j + 1:, j] = 0
    return L, d


def _partial(env, pts, kp, groups, k):  # noqa: F811
    """groups: (ascending members, picks); returns the factor and the builder's log v."""
    torch, sic, pipeline, h = env
    gp = np.concatenate([[0], np.cumsum([len(m) for m, _ in groups])]).astype(np.int64)
    ptr = np.zeros(len(groups) + 1, np.int64)
    hp = pipeline.HostProblem(pts, kp, k, ptr, np.zeros(0, np.int32), gp,
                              members=np.concatenate([m for m, _ in groups]).astype(np.int64))
    b = pipeline.PartialFactorBuilder(h, hp, sic.SIC_FP64)
    sel = np.full((len(groups), k), -1, np.int32)
    for g, (_, p) in enumerate(groups):
        sel[g, :len(p)] = p
    b.sel_idx.copy_(torch.from_numpy(sel.reshape(-1)))
    b.sel_count.copy_(torch.from_numpy(np.array([len(p) for _, p in groups], np.int32)))
    b.logv.zero_()
    b.fill(pipeline.DeviceProblem(hp))
    h.sync()
    return b.col_ptr.cpu().numpy(), b.val.cpu().numpy(), b.logv.cpu().numpy()


def _partial_errors(pts, kp, groups, got):
    cp, val, logv = got
    err, lerr = [], []
    for m, p in groups:
        U = np.sort(np.concatenate([m, p]))[::-1]
        L, d = _ldl(_theta(kp, pts[U]))
        for i in m:
            j = int(np.where(U == i)[0][0])
            x = np.zeros(j + 1, dtype=LD)
            x[j] = 1 / np.sqrt(d[j])
            for r in range(j - 1, -1, -1):
                x[r] = -np.dot(L[r + 1:j + 1, r], x[r + 1:])
            err.append(float(np.abs(val[cp[i]:cp[i + 1]] - x[::-1]).max() / np.abs(x).max()))
            lerr.append(abs(float(logv[i] - np.log(d[j]))))
    return np.array(err), np.array(lerr)


def _groups(n, k, sizes):
    """Disjoint nonadjacent groups over n points, every first member early, picks anywhere after it."""
    order = np.argsort(synthetic.uniform(3, 9, n), kind="stable")
    order = order[order >= len(sizes)]
    out, at = [], 0
    for g, m in enumerate(sizes):
        mem = np.sort(np.concatenate([[g], order[at:at + m - 1]]))
        at += m - 1
        rest = np.setdiff1d(np.arange(g + 1, n), mem)
        out.append((mem, rest[np.argsort(synthetic.uniform(4 + g, 9, len(rest)), kind="stable")][:k]))
    return out


def test_partial_fill(env):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(3, 1, 0.2, 1.0, 1e-2)
    pts = synthetic.points(900, 3, 12)
    groups = _groups(900, 40, [1, 7, 24, 33, 64])  # both size classes
    err, lerr = _partial_errors(pts, kp, groups, _partial(env, pts, kp, groups, 40))
    u = 2.0 ** -53
    assert err.mean() <= 6 * u and lerr.mean() <= 6 * u


def test_partial_fill_with_a_far_point(env):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-2)
    pts = synthetic.points(400, 2, 13)
    groups = _groups(400, 24, [9, 40])
    for m, p in groups:  # the far point is the latest position
        p[:] = np.concatenate([p[p != 399][:23], [399]]) if 399 not in m else p
    pts[399] = FAR
    err, lerr = _partial_errors(pts, kp, groups, _partial(env, pts, kp, groups, 24))
    assert err.max() <= 1e-12 and lerr.max() <= 1e-12


@pytest.mark.parametrize("units", [40, 1800])  # the flat kernel and the panels
def test_side_state_with_a_far_point(env, units):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 5, 0.2, 1.3, 1e-2)
    n, k = 2000, 19
    pts = synthetic.points(n, 2, 14)
    pts[n - 1] = FAR
    targets = (5 * (np.arange(units) % 300)).astype(np.int32)
    sel = np.stack([1500 + (7 * np.arange(k) + 13 * (u % 31)) % 480 for u in range(units)]).astype(np.int32)
    sel[:, -1] = n - 1
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731

    def side(cnt):
        out = [torch.zeros(units * k, dtype=torch.float64, device="cuda") for _ in range(2)]
        sic.side_state_fp64(h, dpts, kp, d(sel.reshape(-1)), d(np.full(units, cnt, np.int32)), k, targets=d(targets),
                            pvar=out[0], pvar_p=out[1])
        h.sync()
        return [x.view(units, k).cpu().numpy()[:, :k - 1] for x in out]

    dpts = d(pts)
    for a, b in zip(side(k), side(k - 1)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_a_point_without_coordinates_has_no_factor(env, value):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-2)
    pts = synthetic.points(200, 2, 15)
    groups = _groups(200, 12, [6])
    pts[groups[0][1][3], 1] = value
    with pytest.raises(sic.SicError) as e:
        _partial(env, pts, kp, groups, 12)
    assert e.value.code == sic.SIC_ERR_NOT_PD
    for units in (20, 1800):
        d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        sel = np.tile(groups[0][1].astype(np.int32), (units, 1))
        out = torch.zeros(units * 12, dtype=torch.float64, device="cuda")
        sic.side_state_fp64(h, d(pts), kp, d(sel.reshape(-1)), d(np.full(units, 12, np.int32)), 12,
                            targets=d(np.zeros(units, np.int32)), pvar=out)
        with pytest.raises(sic.SicError) as e:
            h.sync()
        assert e.value.code == sic.SIC_ERR_NOT_PD
        assert np.all(np.isnan(out.cpu().numpy()))
