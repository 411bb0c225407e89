"""The adjoint rotation at the edges of the rule that picks its kernel (152 SMs):
pairs of CTAs on planes of 88 to 96 with partial tiles, odd counts of angles and
groups of 16 and fewer, and a last group too small for pairs; tiles and columns
at 64 and 65 to 128 along z; z segments in one wave, in a short second wave and
in a fuller one.  Against the same angles back projected one at a time.

Tolerance: the same non-negative float32 terms, up to 9 a sample and angle over
20 angles, in different orders: (9 x 20 + 20) 2^-24 = 1.2e-5 of the value at
worst.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

PAIRS = [(88, 72, 8, 1), (89, 100, 9, 2), (93, 128, 18, 1), (95, 68, 20, 1), (96, 88, 11, 1)]
OTHERS = [(88, 72, 7, 1), (87, 72, 9, 1), (97, 68, 5, 2), (96, 64, 6, 1), (96, 160, 4, 1), (102, 160, 5, 1),
          (121, 160, 3, 1), (128, 40, 4, 2), (136, 64, 5, 1), (137, 64, 5, 1), (128, 32, 4, 1)]


def _tiles(n):
    return ((n + 7) // 8) ** 2


@pytest.mark.parametrize("n,nz,angles,batch", PAIRS + OTHERS)
def test_rule_edges_equal_single_angles(spect_lib, cuda, n, nz, angles, batch):
    if (n, nz, angles, batch) in PAIRS:  # the cases reach the pair kernel
        assert n >= 88 and 64 < nz <= 128 and angles >= 8
        assert _tiles(n) <= torch.cuda.get_device_properties(cuda).multi_processor_count
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
