"""The relative difference prior's gradient on voxels near and below the
smallest normal float, which multiplicative updates leave in air: finite, and
the definition in float64 where every pair's denominator is a normal float.

Tolerance as in test_gpu_prior_shapes.py: 34 roundings of the sum of the
terms' magnitudes.
"""
import numpy as np
import pytest

from test_gpu_prior_shapes import _reference

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TINY = 2.0 ** -126


def _gradient(spect_lib, x):
    t = torch.from_numpy(x).cuda()
    g = torch.full(x.shape, float("nan"), device="cuda")
    spect_lib.spect_prior_grad(t, "rdp", g, delta=1.0, gamma=2.0)
    return g.cpu().numpy()


@pytest.mark.parametrize("value", [1e-37, 1e-38, 1e-39, 1e-40, 1e-45])
def test_equal_voxels(spect_lib, value):
    x = np.full((4, 4, 8), value, dtype=np.float32)
    assert x.max() > 0.0
    assert np.array_equal(_gradient(spect_lib, x), np.zeros_like(x))


@pytest.mark.parametrize("lo,hi", [(-45.0, -36.0), (-45.0, 2.0), (-25.0, -15.0)])
def test_mixed_voxels(spect_lib, lo, hi):
    rng = np.random.Generator(np.random.PCG64(7))
    x = (10.0 ** rng.uniform(lo, hi, size=(6, 6, 12))).astype(np.float32)
    x[rng.uniform(size=x.shape) < 0.3] = 0.0
    g = _gradient(spect_lib, x)
    assert np.all(np.isfinite(g))
    # S >= the sum of the two voxels: voxels of at least TINY have every pair normal
    ref, mag = _reference(x.astype(np.float64), "rdp", 1.0, 2.0)
    normal = x >= TINY
    assert normal.any()
    assert np.all(np.abs(g - ref)[normal] <= 34 * 2.0 ** -24 * mag[normal] + 1e-30)
