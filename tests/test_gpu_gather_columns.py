"""The per-column adjoint rotation on both sides of the launch size that picks
its two variants (16 warps an SM: 2432 on 152 SMs), with several columns to a
warp, one, and two warps to a column, against the same angles back projected
one at a time and summed in float64.

Tolerance: the same non-negative float32 terms, up to 9 a sample and angle over
10 angles, summed in another grouping: (9 x 10 + 10) 2^-24 = 6e-6 of the value
at worst.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,angles,batch", [
    (98, 24, 10, 1), (99, 24, 3, 2),     # four columns a warp: 2401, 2451 warps
    (69, 40, 9, 1), (70, 40, 2, 3),      # two: 2381, 2450
    (49, 68, 7, 2), (50, 72, 10, 1),     # one: 2401, 2500
    (34, 132, 5, 2), (35, 148, 10, 1),   # two warps a column: 2312, 2450
    (3, 4, 4, 1)])
def test_columns_equal_single_angles(spect_lib, cuda, n, nz, angles, batch):
    rng = np.random.Generator(np.random.PCG64(n + nz + angles))
    mu = torch.from_numpy(rng.uniform(0.0, 0.05, size=(n, n, nz)).astype(np.float32)).to(cuda)
    q = torch.from_numpy(rng.uniform(0.1, 2.0, size=(batch, angles, n, nz)).astype(np.float32)).to(cuda)
    whole = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles), mu)
    single = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles, n_subsets=angles), mu)
    got = whole.back(q)
    ref = torch.zeros((batch, n, n, nz), device=cuda, dtype=torch.float64)
    for a in range(angles):
        ref += single.back(q[:, a:a + 1].contiguous(), subset=a).double()
    assert torch.all((got.double() - ref).abs() <= 6e-6 * ref + 1e-30)
    assert float(ref.max()) > 0.0
    for b in range(batch):  # a volume alone: the same bits as in the batch
        assert torch.equal(whole.back(q[b]), got[b])
    whole.check()
    whole.close()
    single.close()
