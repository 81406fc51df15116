"""The double-precision selections (fixed-point factor rows) where the representation or the launch
plan could go wrong: variances far from 1 (the fixed point's exponent), covariances far below its
resolution, non-finite candidates, an odd pick count, and the largest supernode (state mostly in the
workspace).  Picks against the FP64 oracle under the FP64 caps of the parity tests; a power-of-four
scaling of the kernel is exact in every operation, so it must not change a single pick."""
import numpy as np
import pytest

import synthetic
from parity import ReplayStats, replay_multi, replay_single
from test_gpu_parity import CAPS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11648_gb300 import build
    build.build()
    from paper_2307_11648_gb300 import pipeline, sic
    return torch, sic, pipeline, sic.Handle(0)


def _select(env, hp):
    torch, sic, pipeline, h = env
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
    fb.select(pipeline.DeviceProblem(hp))
    h.sync()
    return fb.sel_lists()


@pytest.mark.parametrize("grouped", [False, True])
@pytest.mark.parametrize("var", [4.0 ** -40, 1.9, 4.0 * 1.9, 4.0 ** 60])
def test_variance_scale(env, oracle_lib, grouped, var):
    torch, sic, pipeline, h = env
    base = var
    while base > 2.0:
        base /= 4.0
    while base < 0.5:
        base *= 4.0
    x = synthetic.points(700, 2, 3)
    lists = []
    for v in (base, var):
        kp = sic.kernel(2, 3, 0.1, v, 1e-6 * v)
        hp = (pipeline.prepare_groups(x, kp, 70, 9, mmin=4, mmax=16) if grouped
              else pipeline.prepare_columns(x, kp, 70, 9))
        lists.append(_select(env, hp))
    for a, b in zip(*lists):
        assert a.tolist() == b.tolist()
    okp = oracle_lib.kernel(2, 3, 0.1, var, 1e-6 * var)
    stats = ReplayStats()
    for u in range(0, hp.n_units, 5):
        cand = hp.cand_idx[hp.cand_ptr[u]:hp.cand_ptr[u + 1]]
        if grouped:
            g0, g1 = int(hp.grp_ptr[u]), int(hp.grp_ptr[u + 1])
            replay_multi(oracle_lib, okp, hp.pts, g0, g1 - g0, cand, hp.k, lists[1][u], stats)
        else:
            replay_single(oracle_lib, okp, hp.pts, u, cand, hp.k, lists[1][u], stats)
    stats.check(*CAPS["fp64"])


def test_covariances_below_the_resolution(env, oracle_lib):
    """Length scale 1 / 250 of the spacing: covariances about e^-250 and below."""
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 1, 1e-4, 1.0, 1e-6)
    hp = pipeline.prepare_columns(synthetic.points(300, 2, 5), kp, 40, 6)
    got = _select(env, hp)
    okp = oracle_lib.kernel(2, 1, 1e-4, 1.0, 1e-6)
    for i in range(hp.n):
        cand = hp.cand_idx[hp.cand_ptr[i]:hp.cand_ptr[i + 1]]
        ref = oracle_lib.select_single(okp, hp.pts, i, cand, hp.k)["sel"].tolist() if len(cand) else []
        assert got[i].tolist() == ref, i


@pytest.mark.parametrize("grouped", [False, True])
def test_a_candidate_without_coordinates_is_never_picked(env, grouped):
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-6)
    x = synthetic.points(400, 2, 7)
    hp = pipeline.prepare_groups(x, kp, 50, 12, mmin=4, mmax=16) if grouped else pipeline.prepare_columns(x, kp, 50, 12)
    before = _select(env, hp)
    p = hp.n - 1  # the last position is in the most lists
    users = [u for u in range(hp.n_units) if p in before[u].tolist()]
    assert users
    hp.pts[p] = np.nan
    last = hp.n_units - 1  # the unit that holds the point itself: a supernode has no factor there
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64)
    fb.select(pipeline.DeviceProblem(hp))
    if grouped:
        with pytest.raises(sic.SicError) as e:
            h.sync()
        assert (e.value.code, e.value.unit) == (sic.SIC_ERR_NOT_PD, last)
    else:
        h.sync()
    after = fb.sel_lists()
    for u in range(last):
        assert p not in after[u].tolist()
        if u not in users:
            assert after[u].tolist() == before[u].tolist()


@pytest.mark.parametrize("C,m,k", [(4096, 64, 128), (1023, 63, 63), (513, 1, 127), (33, 5, 40)])
def test_supernode_extremes(env, oracle_lib, C, m, k):
    torch, sic, pipeline, h = env
    kp = sic.kernel(3, 5, 0.4, 1.0, 1e-4)
    okp = oracle_lib.kernel(3, 5, 0.4, 1.0, 1e-4)
    n = C + 2 * m + 7
    P = synthetic.points(n, 3, 9)
    gp = np.array([0, m, 2 * m], np.int64)
    ptr, idx = sic.prep_candidates_groups(P, gp, C)
    hp = pipeline.HostProblem(P, kp, k, ptr, idx, gp)
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64, nnz_cap=1)
    fb.ws_sel.fill_(0xFF)
    fb.select(pipeline.DeviceProblem(hp))
    h.sync()
    stats = ReplayStats()
    for u, sel in enumerate(fb.sel_lists()):
        assert len(sel) == min(k, C)
        replay_multi(oracle_lib, okp, P, u * m, m, idx[ptr[u]:ptr[u + 1]], k, sel, stats)
    stats.check(*CAPS["fp64"])
