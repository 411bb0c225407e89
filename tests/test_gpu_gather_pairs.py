"""The adjoint rotation by pairs of CTAs that share the angles (launches of
fewer tiles than SMs, four angles or more) against the same angles back
projected one at a time, which takes no pairs: odd and even counts of angles,
several groups of 16, planes with partial tiles, columns shorter than a warp's
32 float4 and of odd quarters, and batches.

Tolerance: both sum the same non-negative float32 terms, up to 9 a sample and
angle over 20 angles, in different orders: (9 x 20 + 20) 2^-24 = 1.2e-5 of the
value at worst.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,angles,batch", [(96, 96, 4, 1), (96, 96, 5, 2), (97, 44, 7, 1), (98, 128, 20, 1),
                                               (96, 60, 16, 3), (96, 40, 19, 1)])
def test_pairs_equal_single_angles(spect_lib, cuda, n, nz, angles, batch):
    rng = np.random.Generator(np.random.PCG64(n + nz + angles))
    mu = torch.from_numpy(rng.uniform(0.0, 0.05, size=(n, n, nz)).astype(np.float32)).to(cuda)
    q = torch.from_numpy(rng.uniform(0.1, 2.0, size=(batch, angles, n, nz)).astype(np.float32)).to(cuda)
    whole = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles), mu)
    single = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles, n_subsets=angles), mu)
    got = whole.back(q)
    ref = torch.zeros((batch, n, n, nz), device=cuda, dtype=torch.float64)
    for a in range(angles):
        ref += single.back(q[:, a:a + 1].contiguous(), subset=a).double()
    assert torch.all((got.double() - ref).abs() <= 1.2e-5 * ref + 1e-30)
    assert float(ref.max()) > 0.0
    for b in range(batch):  # a volume alone: the same bits as in the batch
        assert torch.equal(whole.back(q[b]), got[b])
    whole.check()
    whole.close()
    single.close()
