"""The kernel-matrix product's FP32 square root against the library's: bit for bit over every significand at both parities of
the exponent, at random scales from 2^-100 up, and at zero and infinity."""
import numpy as np
import pytest

from test_gpu_parity import env  # noqa: F401

pytestmark = pytest.mark.gpu


def _both(env, x):  # noqa: F811
    torch, sic, _, h = env
    root, ref = sic.selftest_sqrt_f32(h, torch.from_numpy(x).cuda())
    h.sync()
    return root.cpu().numpy(), ref.cpu().numpy()


def test_every_significand(env):  # noqa: F811
    x = np.arange(0x3f800000, 0x40800000, dtype=np.uint32).view(np.float32)  # [1, 4)
    root, ref = _both(env, x)
    assert np.array_equal(root, ref)


def test_scales(env):  # noqa: F811
    r = np.random.RandomState(3)
    bits = (r.randint(27, 255, 1 << 21).astype(np.uint32) << 23) | r.randint(0, 1 << 23, 1 << 21).astype(np.uint32)
    x = np.concatenate([bits.view(np.float32), np.array([0.0, np.inf, 2.0 ** -100], np.float32)])
    root, ref = _both(env, x)
    assert np.array_equal(root, ref)
    tiny = (r.randint(0, 27 << 23, 1 << 16).astype(np.uint32)).view(np.float32)
    root, _ = _both(env, tiny)
    assert np.all((root >= 0) & (root <= np.float32(2.0 ** -49)))
