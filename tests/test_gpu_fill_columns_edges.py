"""The one-warp fill of single columns at the edges of its lanes (picks 1, 31, 32, 33, 48, and 49, which takes the
CTA-wide fill), short columns at the end of the ordering, a slice of columns, and its error reports, against the
oracle with the parity tests' tolerances."""
import numpy as np
import pytest

import synthetic
from parity import column_errors
from test_gpu_parity import L_TOL, LOGV_TOL, _okernel, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 31, 32, 33, 48, 49])
@pytest.mark.parametrize("dim,var", [(2, 1.0), (3, 2.5e-7)])
def test_against_the_oracle(env, oracle_lib, k, dim, var):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(dim, 3, 0.3, var, 1e-6 * var)
    hp = pipeline.prepare_columns(synthetic.points(150, dim, 12), kp, 64, k)
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
    fb.run(pipeline.DeviceProblem(hp))
    h.sync()
    sels = fb.sel_lists()
    cp, ri, val, logv = fb.csc()
    ocp, ori, oval, ologv = oracle_lib.factor_columns(_okernel(oracle_lib, kp), hp.pts, sels)
    assert np.array_equal(cp, ocp) and np.array_equal(ri, ori)
    for i in range(hp.n):
        assert column_errors(val[cp[i]:cp[i + 1]], oval[cp[i]:cp[i + 1]]) <= L_TOL
    assert np.max(np.abs(logv - ologv)) <= LOGV_TOL
    # a slice of the columns gives the same entries
    part = pipeline.slice_problem(hp, 37, 111)
    fs = pipeline.FactorBuilder(h, part, sic.SIC_FP64)
    fs.run(pipeline.DeviceProblem(part))
    h.sync()
    scp, sri, sval, slogv = fs.csc()
    assert np.array_equal(sval, val[cp[37]:cp[111]]) and np.array_equal(sri, ri[cp[37]:cp[111]])
    assert np.array_equal(slogv, logv[37:111])


@pytest.mark.parametrize("what", ["before", "twice", "range", "singular"])
def test_errors(env, what):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.3, 1.0, 0.0 if what == "singular" else 1e-6)
    pts = synthetic.points(80, 2, 12)
    if what == "singular":
        pts[70] = pts[75]
    hp = pipeline.HostProblem(pts, kp, 4, np.zeros(81, np.int64), np.zeros(1, np.int32))
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
    sel = np.full((80, 4), -1, np.int32)
    cnt = np.zeros(80, np.int32)
    sel[3] = [70, 75, 20, 30]
    cnt[3] = 4
    if what == "before":
        sel[3, 1] = 2
    elif what == "twice":
        sel[3, 1] = 70
    elif what == "range":
        sel[3, 1] = 80
    fb.sel_idx.copy_(torch.from_numpy(sel.reshape(-1)))
    fb.sel_count.copy_(torch.from_numpy(cnt))
    fb.fill(pipeline.DeviceProblem(hp))
    with pytest.raises(sic.SicError) as e:
        h.sync()
    assert (e.value.code, e.value.unit) == (sic.SIC_ERR_NOT_PD if what == "singular" else sic.SIC_ERR_INVALID, 3)
