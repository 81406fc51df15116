"""The FP32-mode product with Theta, row by row: a row is as good as its own sum S_i = sum_j |Theta_ij x_j|, whatever the
largest x is -- for dense, sparse and very uneven right-hand sides, and for scales outside FP32's range.

Theta is the product's own, from unit vectors (an FP32 entry times 1 is exact on either path), and is checked against
the Matern function in FP64: coordinates, distance and exponent are FP32 numbers, so an entry is off by
at most (6 + 2 t + 2 c / ell) 2^-23 of itself at t = c r / ell, down to FP32's smallest numbers.

Tolerance of the sums.  Digits: cut at 2^-64 of the largest x and of the variance, levels from 9 on left out, together below
n 2^-63 max|x| of the variance, in rows of S_i >= sqrt(n) 2^-20 of that: sqrt(n) 2^-43 S_i.  Double-FP32: at most
64 terms of 2^-47 each between FP64 additions: 2^-41 S_i.  And the rounding of the FP64 result."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


def _product(env, pts, kp, x):  # noqa: F811
    torch, sic, _, h = env
    y = torch.full(x.shape, 7.0, dtype=torch.float64, device="cuda")
    sic.matern_matvec(h, torch.from_numpy(pts).cuda(), kp, 0.0, sic.SIC_FP32_MIXED,
                      torch.from_numpy(np.ascontiguousarray(x)).cuda(), y)
    h.sync()
    return y.cpu().numpy()


def _theta(env, pts, kp):  # noqa: F811
    n = len(pts)
    K = np.zeros((n, n))
    for j in range(0, n, 8):
        w = min(8, n - j)
        K[:, j:j + w] = _product(env, pts, kp, np.eye(n, dtype=np.float64)[:, j:j + w])
    return K


@pytest.mark.parametrize("dim,nu_x2,ell,n", [(1, 1, 0.01, 200), (2, 3, 0.02, 515), (3, 5, 0.05, 515), (1, 5, 0.3, 129),
                                             (2, 1, 0.3, 200), (3, 3, 0.02, 1031)])
def test_every_row_at_its_own_scale(env, dim, nu_x2, ell, n):  # noqa: F811
    torch, sic, _, h = env
    var = 0.7
    kp = sic.kernel(dim, nu_x2, ell, var, 0.0)
    pts = synthetic.points(n, dim, 8)
    K = _theta(env, pts, kp)
    r = np.sqrt(((pts[:, None] - pts[None]) ** 2).sum(2))
    c = np.sqrt(nu_x2) / ell
    t = c * r
    exact = var * np.exp(-t) * {1: 1 + 0 * t, 3: 1 + t, 5: 1 + t + t * t / 3}[nu_x2]
    assert np.all(np.abs(K - exact) <= exact * (6 + 2 * t + 2 * c) * 2.0 ** -23 + 1e-36)
    assert np.array_equal(K, K.T)

    x = synthetic.normal(3, n * 8).reshape(n, 8)
    x[:, 1] = 0.0
    x[::40, 1] = 1.0                       # sparse
    x[n // 2, 2] = 1e6                     # spikes
    x[n // 3, 3] = 1e16
    x[:, 4] *= np.exp2(-45 * synthetic.uniform(5, 6, n))  # a wide range
    x[:, 5] = 0.0
    x[7, 5] = 1.0                          # a unit vector
    x[:, 6] *= 1e-200                      # beyond FP32
    x[n // 2, 6] = 1e-190
    x[:, 7] *= 1e200
    y = _product(env, pts, kp, x)
    L = np.longdouble
    ref = K.astype(L) @ x.astype(L)
    S = K.astype(L) @ np.abs(x).astype(L)
    err = np.abs(y.astype(L) - ref)
    assert np.all(err <= (np.sqrt(n) * 2.0 ** -43 + 2.0 ** -41) * S + 4e-16 * np.abs(ref))


def test_the_recomputed_rows_use_the_same_theta(env):  # noqa: F811
    """A unit vector, alone and beside a spike at a point without any covariance: the latter's rows are recomputed."""
    torch, sic, _, h = env
    for dim, nu_x2 in [(2, 3), (3, 5), (1, 1)]:
        kp = sic.kernel(dim, nu_x2, 0.2, 1.3, 0.0)
        pts = synthetic.points(300, dim, 8)
        pts[299] = 500.0
        x = np.zeros((300, 2))
        x[3] = 1.0
        x[299, 1] = 1e18
        y = _product(env, pts, kp, x)
        assert np.array_equal(y[:299, 0], y[:299, 1]) and y[299, 1] == 1e18 * np.float64(np.float32(1.3))


@pytest.mark.parametrize("dim,nu_x2,ell", [(2, 3, 0.02), (3, 5, 0.2), (2, 1, 0.05)])
def test_one_right_hand_side_of_many_points(env, dim, nu_x2, ell):  # noqa: F811
    """The CUDA-core sums: the errors of m terms' double-FP32 sum of random signs come to about sqrt(m) 2^-52 of the sum of
    their magnitudes, 2^-48 on average over the rows at m = 256."""
    torch, sic, _, h = env
    n = 12800
    kp = sic.kernel(dim, nu_x2, ell, 1.0, 0.0)
    pts = torch.from_numpy(synthetic.points(n, dim, 8)).cuda()
    K = torch.zeros(n, n, dtype=torch.float32, device="cuda")
    y8 = torch.zeros(n, 8, dtype=torch.float64, device="cuda")
    rows = slice(0, n, 16)
    for j in range(0, n, 8):
        e = torch.zeros(n, 8, dtype=torch.float64, device="cuda")
        e[torch.arange(j, j + 8), torch.arange(8)] = 1.0
        sic.matern_matvec(h, pts, kp, 0.0, sic.SIC_FP32_MIXED, e, y8)
        K[:, j:j + 8] = y8.float()
    x = torch.from_numpy(synthetic.normal(3, n)).cuda()
    y = torch.zeros_like(x)
    sic.matern_matvec(h, pts, kp, 0.0, sic.SIC_FP32_MIXED, x, y)
    h.sync()
    Ks, xl = K[rows].cpu().numpy().astype(np.longdouble), x.cpu().numpy().astype(np.longdouble)
    err = np.abs(y[rows].cpu().numpy().astype(np.longdouble) - Ks @ xl) / (Ks @ np.abs(xl))
    assert err.mean() <= 2.0 ** -48 and err.max() <= 2.0 ** -43


def test_sparse_right_hand_sides_of_many_points(env):  # noqa: F811
    """From 2048 points on no digits are formed for these; zeros, a unit vector, scales beyond FP32."""
    torch, sic, _, h = env
    n = 2100
    kp = sic.kernel(2, 3, 0.1, 0.7, 0.0)
    pts = synthetic.points(n, 2, 8)
    at = np.arange(0, n, 300)
    K = np.zeros((n, len(at)))
    for j in range(0, len(at), 8):
        e = np.zeros((n, min(8, len(at) - j)))
        e[at[j:j + 8], np.arange(e.shape[1])] = 1.0
        K[:, j:j + 8] = _product(env, pts, kp, e)
    x = np.zeros((n, 4))
    x[at[3], 1] = 1.0
    x[at, 2] = 1e-210 * synthetic.normal(3, len(at))
    x[at, 3] = 1e210 * synthetic.normal(4, len(at))
    y = _product(env, pts, kp, x)
    L = np.longdouble
    ref, S = K.astype(L) @ x[at].astype(L), K.astype(L) @ np.abs(x[at]).astype(L)
    assert np.all(y[:, 0] == 0.0) and np.array_equal(y[:, 1], K[:, 3])
    assert np.all(np.abs(y.astype(L) - ref) <= 2.0 ** -41 * S)


def test_a_point_at_infinity(env):  # noqa: F811
    """The exponential kernel is zero at infinite distance: such a point leaves the other rows as they are without it."""
    torch, sic, _, h = env
    kp = sic.kernel(2, 1, 0.2, 1.0, 1e-4)
    pts = synthetic.points(300, 2, 8)
    x = synthetic.normal(3, 900).reshape(300, 3)
    x[5] *= 1e-2
    pts[5, 0] = np.inf
    y = _product(env, pts, kp, x)
    x[5] = 0.0
    pts[5, 0] = 0.5
    ref = _product(env, pts, kp, x)
    rest = np.arange(300) != 5
    assert np.array_equal(y[rest], ref[rest]) and np.all(np.isnan(y[5]))
