"""Directed selection of one target while another stream keeps the SMs busy: its blocks then leave the grid barrier at
very different times, and nothing that a block reads of another may have moved on by then.  The arithmetic does not
depend on timing, so picks and variances are those of the call alone, bit for bit."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(9729, 48), (65536, 24)])
@pytest.mark.parametrize("prec_name", ["fp64", "fp32"])
def test_same_result_beside_other_work(n, k, prec_name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11648_gb300 import build
    build.build()
    from paper_2307_11648_gb300 import sic
    h = sic.Handle(0)
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-4)
    x = synthetic.points(n + 1, 2, 33)
    prec = sic.SIC_FP64 if prec_name == "fp64" else sic.SIC_FP32_MIXED
    train, target = torch.from_numpy(x[1:].copy()).cuda(), torch.from_numpy(x[0].copy()).cuda()
    ws = sic._ws(sic.select_single_workspace(n, k, prec), "cuda")
    out = []
    for rep in range(13):  # the first one alone
        idx = torch.empty(k, dtype=torch.int32, device="cuda")
        var = torch.zeros(k + 1, dtype=torch.float64, device="cuda")
        cnt = torch.empty(1, dtype=torch.int32, device="cuda")
        out.append((idx, var, cnt))
    a = torch.zeros(1 << 22, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for rep, (idx, var, cnt) in enumerate(out):
        if rep:
            with torch.cuda.stream(side):
                for _ in range(40 + 7 * rep):
                    a.mul_(1.0001)
        sic.select_single(h, train, target, kp, k, prec, idx, var, cnt, ws)
        torch.cuda.synchronize()
    h.sync()
    idx, var, cnt = (t.cpu().numpy() for t in out[0])
    assert cnt[0] == k and np.all(np.diff(var) <= 0)
    for o in out[1:]:
        assert all(np.array_equal(r, t.cpu().numpy()) for r, t in zip((idx, var, cnt), o))
