"""The double-precision selections where their fixed-point format runs out.  A candidate far out: coordinates held to
2^-61 of the unit's largest would lose bits of every other distance (2^34 away: 1e-8 of the length scale), FP64
differences lose none, so the decreases stay within rounding (1e-11 at nugget 1e-2) of those without that candidate.
Points many length scales apart on a line: what decides between two of them are products of kernel entries below 2^-58
of the variance; the picks are the FP64 oracle's."""
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


def _line(seed):
    """A target at 0, five points within two length scales of it, then chains to both sides with gaps of 14 .. 40 length
    scales: whether a point behind another one comes before one of the other side depends on the covariance that
    the former leaves it."""
    near = 0.008 * np.arange(1, 6) + 0.003 * synthetic.uniform(seed, 1, 5)
    gaps = 0.28 + 0.5 * synthetic.uniform(seed, 2, 8)
    far = np.concatenate([0.06 + np.cumsum(gaps[:4]), -np.cumsum(gaps[4:])])
    x = np.concatenate([[0.0], np.concatenate([near, far])[np.argsort(synthetic.uniform(seed, 3, 13), kind="stable")]])
    return np.ascontiguousarray(x[:, None])


@pytest.mark.parametrize("nu_x2", [3, 5])
@pytest.mark.parametrize("what", ["columns", "single"])
def test_a_chain_of_distant_points(env, oracle_lib, what, nu_x2):  # noqa: F811
    torch, sic, pipeline, h = env
    kp, okp = sic.kernel(1, nu_x2, 0.02, 1.0, 1e-4), oracle_lib.kernel(1, nu_x2, 0.02, 1.0, 1e-4)
    k = 9
    for seed in range(40):
        pts = _line(seed)
        cand = np.arange(1, 14, dtype=np.int32)
        ref = oracle_lib.select_single(okp, pts, 0, cand, k)["sel"].tolist()
        assert len(ref) > 6  # well into the chain
        if what == "columns":
            hp = pipeline.HostProblem(pts, kp, k, np.array([0, 13], np.int64), cand, None, n_cols=1,
                                      targets=np.zeros(1, np.int32), bounds=(13, 1))
            got = _gains(env, hp)[0]
            got = got[got >= 0].tolist()
        else:
            idx = torch.empty(k, dtype=torch.int32, device="cuda")
            var = torch.zeros(k + 1, dtype=torch.float64, device="cuda")
            cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
            ws = sic._ws(sic.select_single_workspace(13, k, sic.SIC_FP64), "cuda")
            sic.select_single(h, torch.from_numpy(pts[1:].copy()).cuda(), torch.from_numpy(pts[0].copy()).cuda(), kp, k,
                              sic.SIC_FP64, idx, var, cnt, ws)
            h.sync()
            got = (idx.cpu().numpy()[:int(cnt.cpu()[0])] + 1).tolist()
        assert got == ref, seed
