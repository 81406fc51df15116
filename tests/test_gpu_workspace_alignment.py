"""The FP64 supernodal selection takes its workspace at any alignment: its 16-byte loads must not follow the caller's
pointer.  The state of a 1024-candidate supernode lies mostly in the workspace; the picks are those of an aligned one."""
import numpy as np
import pytest

import synthetic
from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [4, 8])
def test_fp64_aggregated(env, offset):  # noqa: F811
    torch, sic, pipeline, h = env
    kp = sic.kernel(2, 3, 0.1, 1.0, 1e-6)
    hp = pipeline.prepare_groups(synthetic.points(1500, 2, 4), kp, 1024, 24, mmin=4, mmax=16)
    dp = pipeline.DeviceProblem(hp)
    fb = pipeline.FactorBuilder(h, hp, sic.SIC_FP64, nnz_cap=1)
    need = sic.select_aggregated_workspace(h, hp.n_units, hp.max_cand, hp.max_m, hp.k, sic.SIC_FP64)
    assert need > 16
    fb.select(dp)
    h.sync()
    ref = fb.sel_idx.cpu().numpy()
    room = torch.full((need + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    fb.ws_sel = room[offset:offset + need]  # exactly what the query asks for
    assert fb.ws_sel.data_ptr() % 16 == offset
    fb.sel_idx.fill_(-7)
    fb.select(dp)
    h.sync()
    assert np.array_equal(fb.sel_idx.cpu().numpy(), ref)
    guard = room.cpu().numpy()
    assert np.all(guard[:offset] == 0xA5) and np.all(guard[offset + need:] == 0xA5)
