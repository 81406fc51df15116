"""Partial selection's two size classes (groups whose state fits an SM twice, and the others) give the same
picks and decreases, bit for bit: the classes' border follows the bound on the candidates, so that a larger bound moves
groups from one class's kernel to the other's.  An invalid group is reported once, whichever class comes first."""
import numpy as np
import pytest

import synthetic
from test_gpu_partial import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name,C,k,bounds", [("fp32", 256, 64, (256, 300, 330)), ("fp32", 40, 16, (40, 560)),
                                                  ("fp64", 96, 48, (96, 150))])
def test_the_border_moves_nothing(env, prec_name, C, k, bounds):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.05, 1.0, 1e-6)
    hp = pipeline.prepare_partial(synthetic.points(4096, 2, 3), kp, C, k)
    b = pipeline.PartialFactorBuilder(h, hp, sic.SIC_FP64 if prec_name == "fp64" else sic.SIC_FP32_MIXED)
    dp = pipeline.DeviceProblem(hp)
    gain = torch.zeros(hp.n_units * k, dtype=torch.float64, device="cuda")
    got = []
    for bound in bounds:
        b.sel_idx.fill_(-7)
        b.sel_count.fill_(-7)
        gain.zero_()
        sic.select_partial(h, dp.pts, hp.kp, dp.grp_ptr, dp.members, dp.cand_ptr, dp.cand_idx, bound, hp.max_m, k,
                           b.prec, b.sel_idx, b.sel_count, gain=gain)
        h.sync()
        got.append((b.sel_idx.cpu().numpy().copy(), b.sel_count.cpu().numpy().copy(), gain.cpu().numpy().copy()))
    assert got[0][1].min() >= 0 and got[0][1].max() == k
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)


def test_invalid_group(env):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.05, 1.0, 1e-6)
    hp = pipeline.prepare_partial(synthetic.points(2048, 2, 3), kp, 64, 16)
    b = pipeline.PartialFactorBuilder(h, hp, sic.SIC_FP32_MIXED)
    dp = pipeline.DeviceProblem(hp)
    m = np.diff(hp.grp_ptr)
    assert m.max() == hp.max_m and (m == hp.max_m).sum() < len(m)
    sic.select_partial(h, dp.pts, hp.kp, dp.grp_ptr, dp.members, dp.cand_ptr, dp.cand_idx, hp.max_cand,
                       int(hp.max_m) - 1, 16, b.prec, b.sel_idx, b.sel_count)
    with pytest.raises(sic.SicError) as e:
        h.sync()
    assert e.value.code == sic.SIC_ERR_INVALID and m[e.value.unit] == hp.max_m
    cnt = b.sel_count.cpu().numpy()
    assert np.all(cnt[m == hp.max_m] == 0) and np.all(cnt[m < hp.max_m] >= 0)
