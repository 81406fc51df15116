"""The side state of many units (panels, two size classes) against the same units in calls of a few (the flat kernel):
unit sizes around the classes' border, picks before and after the targets, counts from 0 to k."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,nu_x2,k", [(2, 3, 8), (3, 5, 33)])
def test_many_units_against_few(env, dim, nu_x2, k):  # noqa: F811
    torch, sic, pipeline, h = env
    units = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    m = np.where(np.arange(units) % 97 == 0, 1 + np.arange(units) % 64, 1 + np.arange(units) % 3)
    m[:4] = 31, 32, 33, 64
    gp = np.concatenate([[0], np.cumsum(m)]).astype(np.int64)
    n = int(gp[-1])
    kp = sic.kernel(dim, nu_x2, 0.1, 1.0, 1e-4)
    pts = synthetic.points(n, dim, 6)
    cnt = (np.arange(units) % (k + 1)).astype(np.int32)
    sel = np.full((units, k), -1, np.int32)
    for u in range(units):  # any points but the unit's own
        p = (gp[u] + m[u] + 7 * np.arange(cnt[u]) + 11 * (u % 13)) % n
        inside = (p >= gp[u]) & (p < gp[u] + m[u])
        cnt[u] = (~inside).sum()
        sel[u, :cnt[u]] = p[~inside]

    def side(lo, hi):
        d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        out = [torch.full(((hi - lo) * k,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
        sic.side_state_fp64(h, d(pts), kp, d(sel[lo:hi].reshape(-1)), d(cnt[lo:hi]), k, grp_ptr=d(gp[lo:hi + 1]), max_m=64,
                            pvar=out[0], pvar_p=out[1], gain=out[2])
        h.sync()
        return [x.cpu().numpy() for x in out]

    many = side(0, units)
    few = [np.concatenate(x) for x in zip(*[side(a, min(a + 500, units)) for a in range(0, units, 500)])]
    # pivots at nugget 1e-4: both factorisations are backward stable, some 1e-16 / 1e-4 relative with a factor for the order
    for a, b in zip(many[:2], few[:2]):
        assert np.max(np.abs(a / b - 1)) <= 1e-9
    assert np.max(np.abs(many[2] - few[2])) <= 2e-9
