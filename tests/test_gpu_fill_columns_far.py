"""Single columns of points many length scales apart: kernel entries far below the fixed point's 2^-60 of the variance.
Each entry of a column is good at its own scale, against NumPy's long double (128 bits where this runs).

Tolerance.  A column is A^-1 e_i over its set, scaled; with Theta's entries and every step good to a few ulp, its error
is at most a few n ulp (n <= 41, together below 1e-13) of the same sum over all elimination paths taken without signs:
the column H^-1 e_i of A's comparison matrix H = diag(A) - |A - diag(A)|, under the same scaling."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401
from test_gpu_unit_precision import _ldl, _theta

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [5, 32, 40])
@pytest.mark.parametrize("nu_x2,ell", [(1, 0.02), (3, 0.01), (5, 0.012)])
def test_entries_at_their_own_scale(env, nu_x2, ell, k):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(3, nu_x2, ell, 1.3, 1e-2)
    n = 90
    g = np.stack(np.meshgrid(np.arange(5), np.arange(5), np.arange(5), indexing="ij"), -1).reshape(-1, 3)
    pts = (0.3 * g + 0.05 * synthetic.uniform(7, 1, 375).reshape(125, 3))[np.argsort(synthetic.uniform(8, 2, 125))][:n]
    pts = np.ascontiguousarray(pts)
    hp = pipeline.HostProblem(pts, kp, k, np.zeros(n + 1, np.int64), np.zeros(1, np.int32))
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
    sel = np.full((n, k), -1, np.int32)
    cnt = np.minimum(k, n - 1 - np.arange(n)).astype(np.int32)
    for i in range(n):
        rest = np.arange(i + 1, n)
        sel[i, :cnt[i]] = rest[np.argsort(synthetic.uniform(i, 3, len(rest)), kind="stable")][:cnt[i]]
    fb.sel_idx.copy_(torch.from_numpy(sel.reshape(-1)))
    fb.sel_count.copy_(torch.from_numpy(cnt))
    fb.fill(pipeline.DeviceProblem(hp))
    h.sync()
    cp, ri, val, logv = fb.csc()
    for i in range(0, n, 3):
        U = np.sort(np.concatenate([[i], sel[i, :cnt[i]]]))[::-1]
        L, d = _ldl(_theta(kp, pts[U]))
        j = len(U) - 1
        x = np.zeros(j + 1, dtype=np.longdouble)
        x[j] = 1 / np.sqrt(d[j])
        for r in range(j - 1, -1, -1):
            x[r] = -np.dot(L[r + 1:j + 1, r], x[r + 1:])
        A = _theta(kp, pts[U])
        Lh, dh = _ldl(2 * np.diag(np.diag(A)) - A)
        y = np.zeros(j + 1, dtype=np.longdouble)  # H^-1 e_i
        y[j] = 1 / dh[j]
        for r in range(j - 1, -1, -1):
            y[r] = -np.dot(Lh[r + 1:j + 1, r], y[r + 1:])
        assert np.all(y >= 0)
        got = val[cp[i]:cp[i + 1]].astype(np.longdouble)[::-1]
        assert np.all(np.abs(got - x) <= 1e-13 * y * np.sqrt(d[j])), i
        assert abs(float(logv[i] - np.log(d[j]))) <= 1e-15
