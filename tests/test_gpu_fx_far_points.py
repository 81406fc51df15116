"""The double-precision selections where their fixed-point format runs out.  A candidate far out: coordinates held to
2^-61 of the unit's largest would lose bits of every other distance (2^34 away: 1e-8 of the length scale), FP64
differences lose none, so the decreases stay within rounding (1e-11 at nugget 1e-2) of those without that candidate."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu
FAR = float(2 ** 34)


def _gains(env, hp):  # noqa: F811
    torch, sic, pipeline, h = env
    b = pipeline.FactorBuilder(h, hp, sic.SIC_FP64, nnz_cap=1, budget=1)
    b.gain.zero_()
    b.select_local(pipeline.DeviceProblem(hp))
    h.sync()
    return b.sel_idx.cpu().numpy(), b.gain.cpu().numpy()


@pytest.mark.parametrize("grouped", [False, True])
def test_a_far_candidate(env, grouped):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 5, 0.2, 1.0, 1e-2)
    n, k, m, units = 1200, 12, (5 if grouped else 1), 60
    pts = synthetic.points(n, 2, 41)
    pts[n - 1] = FAR
    gp = (m * np.arange(units + 1)).astype(np.int64)
    lists = [400 + (np.arange(150) * 5 + 3 * u) % 790 for u in range(units)]

    def problem(extra):
        idx = np.concatenate([np.concatenate([x, extra]) for x in lists]).astype(np.int32)
        ptr = (np.arange(units + 1) * (150 + len(extra))).astype(np.int64)
        if grouped:
            return pipeline.HostProblem(pts, kp, k, ptr, idx, gp, n_cols=int(gp[-1]), bounds=(150 + len(extra), m))
        return pipeline.HostProblem(pts, kp, k, ptr, idx, None, n_cols=units, targets=np.arange(units, dtype=np.int32),
                                    bounds=(150 + len(extra), 1))

    sel, gain = _gains(env, problem([]))
    sel_far, gain_far = _gains(env, problem([n - 1]))
    assert np.array_equal(sel, sel_far)
    assert np.all(gain > 0) and np.max(np.abs(gain - gain_far)) <= 1e-11
