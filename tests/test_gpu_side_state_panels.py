"""The FP64 side state by panels (many units of many picks): both size classes of units against the same units in calls of a
few, which the flat kernel takes; a point far out as the last pick changes no bit before it; coincident points without a
nugget and points without coordinates are reported.  Tolerance of the comparison: both factorisations are backward stable,
some 1e-16 / nugget relative with a factor for the order."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu
K = 44


def _call(env, pts, kp, gp, sel, cnt, max_m):  # noqa: F811
    torch, sic, _, h = env
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    out = [torch.full((len(cnt) * K,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
    sic.side_state_fp64(h, d(pts), kp, d(sel.reshape(-1)), d(cnt), K, grp_ptr=d(gp), max_m=max_m, pvar=out[0],
                        pvar_p=out[1], gain=out[2])
    h.sync()
    return [x.view(-1, K).cpu().numpy() for x in out]


def _units(env, far=False):  # noqa: F811
    torch = env[0]
    units = 10 * torch.cuda.get_device_properties(0).multi_processor_count
    m = np.where(np.arange(units) % 97 == 0, 1 + np.arange(units) % 64, 1 + np.arange(units) % 3)
    m[:4] = 31, 32, 33, 64
    gp = np.concatenate([[0], np.cumsum(m)]).astype(np.int64)
    n = int(gp[-1]) + 1
    pts = synthetic.points(n, 2, 6)
    cnt = (K - np.arange(units) % 7).astype(np.int32)
    sel = np.full((units, K), -1, np.int32)
    for u in range(units):
        p = (gp[u] + m[u] + 7 * np.arange(cnt[u]) + 11 * (u % 13)) % (n - 1)
        p = p[(p < gp[u]) | (p >= gp[u] + m[u])]
        cnt[u] = len(p)
        sel[u, :cnt[u]] = p
    return pts, gp, sel, cnt


def test_against_the_flat_kernel(env):  # noqa: F811
    torch, sic, _, h = env
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-4)
    pts, gp, sel, cnt = _units(env)
    units = len(cnt)
    many = _call(env, pts, kp, gp, sel, cnt, 64)
    few = [np.concatenate(x) for x in zip(*[_call(env, pts, kp, gp[a:a + 501], sel[a:a + 500], cnt[a:a + 500], 64)
                                            for a in range(0, units, 500)])]
    for a, b in zip(many[:2], few[:2]):
        assert np.max(np.abs(a / b - 1)) <= 1e-9
    assert np.max(np.abs(many[2] - few[2])) <= 2e-9


def test_a_far_point(env):  # noqa: F811
    torch, sic, _, h = env
    kp = sic.kernel(2, 5, 0.2, 1.3, 1e-2)
    pts, gp, sel, cnt = _units(env)
    pts[-1] = 2.0 ** 34
    before = _call(env, pts, kp, gp, sel, cnt - 1, 64)
    sel[np.arange(len(cnt)), cnt - 1] = len(pts) - 1
    after = _call(env, pts, kp, gp, sel, cnt, 64)
    same = np.arange(K)[None, :] < (cnt - 1)[:, None]
    for a, b in zip(before[:2], after[:2]):
        assert np.array_equal(a[same], b[same])


@pytest.mark.parametrize("what", ["coincident", "nan", "inf"])
def test_reports(env, what):  # noqa: F811
    torch, sic, _, h = env
    pts, gp, sel, cnt = _units(env)
    units = len(cnt)
    for u in (0, 5, units - 1):
        bad = pts.copy()
        if what == "coincident":
            bad[sel[u, 7]] = bad[sel[u, 3]]
        else:
            bad[sel[u, 7], 1] = np.nan if what == "nan" else np.inf
        kp = sic.kernel(2, 3, 0.1, 1.3, 0.0 if what == "coincident" else 1e-2)
        with pytest.raises(sic.SicError) as e:
            _call(env, bad, kp, gp, sel, cnt, 64)
        assert e.value.code == sic.SIC_ERR_NOT_PD
