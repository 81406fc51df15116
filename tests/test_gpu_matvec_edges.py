"""The FP32-mode product with Theta at the edges of its row tiles, source chunks and cluster shares, against the
exact sum of the kernel entries that the product itself returns for unit vectors.  Tolerance: the digits left
out are below 2^-46 max|x| of the variance per term (x and Theta each to 2^-47, levels from 6 on), so
n 2^-45 variance max|x| bounds a row's error, plus the rounding of the FP64 result."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11648_gb300 import build
    build.build()
    from paper_2307_11648_gb300 import sic
    return torch, sic, sic.Handle(0)


def _product(env, pts, kp, x):
    torch, sic, h = env
    y = torch.full(x.shape, float("nan"), dtype=torch.float64, device="cuda")
    sic.matern_matvec(h, torch.from_numpy(pts).cuda(), kp, 1e-3, sic.SIC_FP32_MIXED, torch.from_numpy(x).cuda(), y)
    h.sync()
    return y.cpu().numpy()


@pytest.mark.parametrize("n,nrhs,dim,nu_x2,var", [(1, 1, 2, 3, 1.0), (127, 3, 1, 1, 0.3), (128, 8, 2, 3, 4.0),
                                                  (129, 1, 3, 5, 1.0), (515, 5, 3, 5, 3.7), (2049, 8, 2, 3, 1.0)])
def test_against_the_exact_sum(env, n, nrhs, dim, nu_x2, var):
    torch, sic, h = env
    kp = sic.kernel(dim, nu_x2, 0.3, var, 1e-4)
    pts = synthetic.points(n, dim, 8)
    K = np.zeros((n, n))
    for j in range(0, n, 8):
        w = min(8, n - j)
        K[:, j:j + w] = _product(env, pts, kp, np.eye(n, dtype=np.float64)[:, j:j + w].copy())
    x = synthetic.normal(3, n * nrhs).reshape(n, nrhs)
    x[n // 2, 0] = 1e6  # one right-hand side with a wide range
    x[:, nrhs - 1] *= 1e-200
    got = _product(env, pts, kp, x)
    ref = (K.astype(np.longdouble) @ x.astype(np.longdouble)).astype(np.float64)
    tol = n * 2.0 ** -45 * var * np.abs(x).max(axis=0) + 4e-16 * np.abs(ref)
    assert np.all(np.abs(got - ref) <= tol)


def test_zeros_and_non_finite_values(env):
    torch, sic, h = env
    kp = sic.kernel(2, 3, 0.3, 1.0, 1e-4)
    n = 300
    pts = synthetic.points(n, 2, 8)
    x = synthetic.normal(3, n * 4).reshape(n, 4)
    x[:, 1] = 0.0
    x[17, 2] = np.inf
    y = _product(env, pts, kp, x)
    assert np.all(np.isfinite(y[:, [0, 3]])) and np.all(y[:, 1] == 0.0) and not np.any(np.isfinite(y[:, 2]))
    pts[5] = np.nan
    assert not np.any(np.isfinite(_product(env, pts, kp, x)[:, 0]))


def test_both_kernels_agree(env):
    """One right-hand side at a size that takes the CUDA-core sums against the same one among three."""
    torch, sic, h = env
    kp = sic.kernel(2, 3, 0.05, 1.0, 1e-4)
    n = 12289
    pts = synthetic.points(n, 2, 8)
    x = synthetic.normal(3, n * 3).reshape(n, 3)
    one, three = _product(env, pts, kp, x[:, 0].copy()), _product(env, pts, kp, x)
    assert np.max(np.abs(one - three[:, 0])) <= n * 2.0 ** -45 * np.abs(x).max()
