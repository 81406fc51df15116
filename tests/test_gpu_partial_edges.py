"""Partial selection where its launch could go wrong: column counts across the hand-over chunks (16), the
first warp's blocks of pivot rows (32) and its last block size (up to 191 columns), more candidate rows
than walking threads, one target, fewer candidates than picks.  Replayed by the oracle with the
tolerances of tests/test_gpu_partial.py."""
import numpy as np
import pytest

import synthetic
from parity import ReplayStats
from test_gpu_partial import _okernel, _replay_partial, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec_name,m,C,k", [("fp32", 64, 130, 127), ("fp32", 1, 1000, 20), ("fp32", 17, 10, 16),
                                             ("fp64", 33, 60, 60), ("fp64", 2, 600, 17)])
def test_shapes(env, oracle_lib, prec_name, m, C, k):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.15, 1.0, 1e-4)
    okp = _okernel(oracle_lib, kp)
    n, groups = C + m + 200, 2
    P = synthetic.points(n, 2, 17)
    members, cand = [], []
    for g in range(groups):
        order = np.argsort(synthetic.uniform(40 + g, 5, n), kind="stable")
        mem = np.sort(order[:m])
        mem[0] = g  # an early first member: nearly every other point may be a candidate
        rest = np.setdiff1d(np.arange(g + 1, n), mem)
        members.append(np.unique(mem))
        cand.append(rest[np.argsort(synthetic.uniform(50 + g, 5, len(rest)), kind="stable")][:C].astype(np.int32))
    gp = np.concatenate([[0], np.cumsum([len(x) for x in members])]).astype(np.int64)
    ptr = np.arange(groups + 1, dtype=np.int64) * C
    hp = pipeline.HostProblem(P, kp, k, ptr, np.concatenate(cand), gp, members=np.concatenate(members).astype(np.int64))
    b = pipeline.PartialFactorBuilder(h, hp, sic.SIC_FP64 if prec_name == "fp64" else sic.SIC_FP32_MIXED)
    b.select(pipeline.DeviceProblem(hp))
    h.sync()
    stats = ReplayStats()
    for g, sel in enumerate(b.sel_lists()):
        assert len(sel) == min(k, C)
        _replay_partial(oracle_lib, okp, hp, g, sel, stats, prec_name == "fp32")
    assert stats.frac <= (1e-3 if prec_name == "fp64" else 0.05)
