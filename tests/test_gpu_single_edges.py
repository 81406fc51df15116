"""Directed selection of one target at the edges of its grid: one row, one block (64 rows), the first
row of a second block, rows per block 128 and 256, and rows strided beyond the grid; by oracle
replay under the caps of the directed test (near-ties only in FP64)."""
import numpy as np
import pytest

import synthetic
from parity import ReplayStats, replay_single
from test_gpu_parity import CAPS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(1, 3), (64, 20), (65, 65), (130, 8), (9729, 6), (20001, 5), (80001, 4)])
@pytest.mark.parametrize("prec_name", ["fp64", "fp32"])
def test_grid_edges(oracle_lib, n, k, prec_name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11648_gb300 import build
    build.build()
    from paper_2307_11648_gb300 import sic
    oracle = oracle_lib
    h = sic.Handle(0)
    kp = sic.kernel(2, 3, 0.3, 1.0, 1e-4)
    okp = oracle.kernel(2, 3, 0.3, 1.0, 1e-4)
    x = synthetic.points(n + 1, 2, 31)
    prec = sic.SIC_FP64 if prec_name == "fp64" else sic.SIC_FP32_MIXED
    ws = sic._ws(sic.select_single_workspace(n, k, prec), "cuda")
    ws.fill_(0xFF)  # NaN everywhere: nothing may be read before it is written
    idx = torch.empty(k, dtype=torch.int32, device="cuda")
    var = torch.zeros(k + 1, dtype=torch.float64, device="cuda")
    cnt = torch.empty(1, dtype=torch.int32, device="cuda")
    sic.select_single(h, torch.from_numpy(x[1:].copy()).cuda(), torch.from_numpy(x[0].copy()).cuda(), kp, k, prec,
                      idx, var, cnt, ws)
    h.sync()
    c = int(cnt.cpu()[0])
    sel = idx.cpu().numpy()
    assert c == min(n, k) and np.all(sel[c:] == -1)
    stats = ReplayStats()
    cand = np.arange(1, n + 1, dtype=np.int32)
    replay_single(oracle, okp, x, 0, cand, k, sel[:c] + 1, stats, fp32=prec_name == "fp32")
    stats.check(*(CAPS["fp64"] if prec_name == "fp64" else CAPS["directed_fp32"]))
    if prec_name == "fp64":
        r = oracle.select_single(okp, x, 0, cand, k, forced=sel[:c].tolist())
        assert np.allclose(var.cpu().numpy()[:c + 1], r["vtar"], rtol=1e-8)
