"""The BF16 training step at the edges of its 128-row tiles, of the 152-CTA grid and of the 512-row
chunks of the bias sums, against FP64 backpropagation with the operands rounded where the step
rounds them (W, X, H1, dZ1, dZ2 as operands of the products).

Tolerance: what remains are FP32 sums (relative 2^-24 per term, at most 1e-5 of a sum here) and
values that land on the other side of a BF16 rounding because of them (2^-9 of single terms, whose
share of a gradient's norm stays below 2^-9); 2^-9 of each parameter block's norm bounds both, and a
lost or doubled row moves a block by about 1 / rows of it at the small sizes."""
import numpy as np
import pytest

import synthetic
from oracle import learned as OL

pytestmark = pytest.mark.gpu

BLOCKS = {"W1": (0, 1024), "b1": (1024, 1152), "W2": (1152, 17536), "b2": (17536, 17664), "w3": (17664, 17792),
          "b3": (17792, 17793)}


def _bf16(x):
    import torch
    return torch.from_numpy(np.asarray(x, np.float64)).to(torch.bfloat16).to(torch.float64).numpy()


def _reference(P, X, y, pw):
    d = OL.unpack(P)
    Z1 = X @ d["W1"] + d["b1"]
    H1 = _bf16(OL.gelu(Z1))
    Z2 = H1 @ d["W2"] + d["b2"]
    H2 = OL.gelu(Z2)
    s = H2 @ d["w3"] + d["b3"]
    sig = 1.0 / (1.0 + np.exp(-s))
    dS = (pw * y * (sig - 1.0) + (1 - y) * sig) / len(X)
    dZ2 = np.outer(dS, d["w3"]) * OL.dgelu(Z2)
    dZ1 = (_bf16(dZ2) @ d["W2"].T) * OL.dgelu(Z1)
    g = dict(w3=H2.T @ dS, b3=np.array(dS.sum()), W2=H1.T @ _bf16(dZ2), b2=dZ2.sum(0), W1=X.T @ _bf16(dZ1),
             b1=dZ1.sum(0))
    return OL.pack(g), float(np.mean(pw * y * OL.softplus(-s) + (1 - y) * OL.softplus(s))), s


@pytest.mark.parametrize("batch", [1, 127, 128, 129, 513, 152 * 128 + 1])
def test_bf16_step_at_tile_edges(batch):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2307_11648_gb300 import build
    build.build()
    from paper_2307_11648_gb300 import learned, sic
    h = sic.Handle(0)
    X = synthetic.normal(5, batch * 8).reshape(batch, 8).astype(np.float32)
    y = (synthetic.uniform(6, 3, batch) < 0.3).astype(np.float32)
    P = learned.init_params(3)
    P[1024:1152] = 0.05
    P[17536:17664] = -0.02
    P[17792] = -1.0
    dev = [torch.from_numpy(a).cuda() for a in (P, X, y)]
    g = torch.full((P.size,), float("nan"), dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    score = torch.zeros(batch, dtype=torch.float32, device="cuda")
    ws = sic._ws(sic.mlp_train_workspace(batch), "cuda")
    ws.fill_(0xFF)  # NaN everywhere: nothing may be read before it is written
    sic.mlp_grads(h, *dev, 2.0, True, g, loss, ws, score=score)
    h.sync()
    ref, ref_loss, ref_s = _reference(_bf16(P), _bf16(X), y.astype(np.float64), 2.0)
    got = g.cpu().numpy().astype(np.float64)
    for name, (a, b) in BLOCKS.items():
        err = np.linalg.norm(got[a:b] - ref[a:b]) / np.linalg.norm(ref[a:b])
        assert err <= 2.0 ** -9, (name, err)
    assert float(loss.cpu()[0]) == pytest.approx(ref_loss, rel=2.0 ** -9)
    assert np.allclose(score.cpu().numpy(), ref_s, rtol=0, atol=2.0 ** -9 * np.abs(ref_s).max())
