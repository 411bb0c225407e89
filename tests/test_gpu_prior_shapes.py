"""The prior gradient where its runs along the first axis, its blocks of 32 x 8
voxels and the volume's faces meet, with zeros and values over many orders of
magnitude, against the definition in float64.

Tolerance: a term is a handful of float32 roundings (at most 8) of factors
without cancellation, and up to 26 of either sign are added: 34 x 2^-24 of the
sum of their magnitudes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _reference(x, prior, delta, gamma):
    g, mag = np.zeros_like(x), np.zeros_like(x)
    for di in (-1, 0, 1):
        for dj in (-1, 0, 1):
            for dk in (-1, 0, 1):
                if not (di or dj or dk):
                    continue
                sl = [(slice(max(0, -o), m - max(0, o)), slice(max(0, o), m - max(0, -o)))
                      for o, m in zip((di, dj, dk), x.shape)]
                here, there = tuple(s[0] for s in sl), tuple(s[1] for s in sl)
                a, b = x[here], x[there]
                d = a - b
                if prior == "quadratic":
                    t = d / (2.0 * delta ** 2)
                else:
                    den = a + b + gamma * np.abs(d)
                    t = np.divide(d * (a + 3 * b + gamma * np.abs(d)), den ** 2, out=np.zeros_like(d), where=den > 0)
                t = 2.0 / np.sqrt(di * di + dj * dj + dk * dk) * t
                g[here] += t
                mag[here] += np.abs(t)
    return g, mag


@pytest.mark.parametrize("prior", ["quadratic", "rdp"])
@pytest.mark.parametrize("n,nz", [(1, 1), (1, 5), (2, 4), (4, 33), (5, 32), (9, 36), (17, 65)])
def test_prior_gradient_shapes(spect_lib, cuda, n, nz, prior):
    rng = np.random.Generator(np.random.PCG64(100 * n + nz))
    x = (10.0 ** rng.uniform(-6.0, 4.0, size=(n, n, nz))).astype(np.float32)
    x[rng.uniform(size=x.shape) < 0.3] = 0.0
    g = torch.full(x.shape, float("nan"), device=cuda)
    spect_lib.spect_prior_grad(torch.from_numpy(x).to(cuda), prior, g, delta=0.7, gamma=2.0)
    ref, mag = _reference(x.astype(np.float64), prior, float(np.float32(0.7)), 2.0)
    assert np.all(np.abs(g.cpu().numpy() - ref) <= 34 * 2.0 ** -24 * mag + 1e-30)
