"""Partial selection of many groups (two size classes, two groups per SM for the smaller ones) against the same groups in
calls of a hundred (one class): the same picks and decreases, bit for bit, in both precisions."""
import numpy as np
import pytest

import synthetic
from test_gpu_partial import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name,n,C,k", [("fp32", 4096, 256, 40), ("fp64", 18000, 100, 12)])
def test_many_groups_against_few(env, prec_name, n, C, k):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.05, 1.0, 1e-6)
    hp = pipeline.prepare_partial(synthetic.points(n, 2, 3), kp, C, k)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    prec = sic.SIC_FP64 if prec_name == "fp64" else sic.SIC_FP32_MIXED
    assert hp.n_units > (5 if prec_name == "fp64" else 1) * sms
    dp = pipeline.DeviceProblem(hp)

    def select(lo, hi):
        sel = torch.full(((hi - lo) * k,), -7, dtype=torch.int32, device="cuda")
        cnt = torch.full((hi - lo,), -7, dtype=torch.int32, device="cuda")
        gain = torch.zeros((hi - lo) * k, dtype=torch.float64, device="cuda")
        sic.select_partial(h, dp.pts, hp.kp, dp.grp_ptr[lo:hi + 1].contiguous(), dp.members,
                           dp.cand_ptr[lo:hi + 1].contiguous(), dp.cand_idx, hp.max_cand, hp.max_m, k, prec, sel, cnt,
                           gain=gain)
        h.sync()
        return [x.cpu().numpy() for x in (sel, cnt, gain)]

    many = select(0, hp.n_units)
    few = [np.concatenate(x) for x in zip(*[select(a, min(a + 100, hp.n_units)) for a in range(0, hp.n_units, 100)])]
    assert many[1].min() >= 0
    for a, b in zip(many, few):
        assert np.array_equal(a, b)
