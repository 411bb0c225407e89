"""Whole projections of short planes, which take CTAs of a thread per blur strip,
against the same angles projected one at a time, which do not: one and several
strips to a warp, planes that are no multiple of 16, a field-of-view mask, no
attenuation, more chunks' partials than one launch holds, and batches (one that
takes such CTAs where a volume alone does not).

Tolerance: a bin is the sum of n non-negative float32 terms over depth, in
other groupings on the two sides: 2 n 2^-24 of its value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,angles,batch,kw", [
    (48, 24, 96, 2, {}), (33, 28, 60, 1, {}), (64, 24, 48, 4, {"fov": True}), (57, 36, 40, 1, {}),
    (96, 36, 64, 2, {}), (40, 96, 50, 1, {"attenuation": False}), (32, 24, 300, 3, {}), (32, 36, 17, 4, {}), (20, 4, 64, 1, {}),
    (80, 20, 33, 1, {"psf": False})])
def test_whole_equals_single_angles(spect_lib, cuda, n, nz, angles, batch, kw):
    kw = dict(kw)
    rng = np.random.Generator(np.random.PCG64(n + nz + angles))
    if kw.pop("fov", False):
        kw["fov_mask"] = rng.uniform(0.2, 1.0, size=(angles, n, nz)).astype(np.float32)
    mu = None
    if kw.get("attenuation", True):
        mu = torch.from_numpy(rng.uniform(0.0, 0.05, size=(n, n, nz)).astype(np.float32)).to(cuda)
    x = torch.from_numpy(rng.uniform(0.1, 2.0, size=(batch, n, n, nz)).astype(np.float32)).to(cuda)
    whole = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles, **kw), mu)
    single = spect_lib.Plan(spect_lib.Geometry(n=n, nz=nz, n_angles=angles, n_subsets=angles, **kw), mu)
    got = whole.forward(x).reshape(batch, angles, n, nz)
    for a in range(angles):
        ref = single.forward(x, subset=a).reshape(batch, n, nz).double()
        assert torch.all((got[:, a].double() - ref).abs() <= 2 * n * 2.0 ** -24 * ref + 1e-30), a
    assert float(got.min()) >= 0.0 and float(got.max()) > 0.0
    for b in range(batch):  # a volume alone: the same bits as in the batch
        assert torch.equal(whole.forward(x[b]).reshape(angles, n, nz), got[b])
    whole.check()
    whole.close()
    single.close()
