"""The quad walk of the listmode PET projector against the walk of the image
that calls with few lines take, on the same lines: grids with single-voxel
and odd axes, lines along every principal axis, axis-parallel, on ties,
ending inside the image, missing it and degenerate, with and without time of
flight.  A call with at least one line per 32 voxels walks quads; the same
lines in short calls walk the image.

Tolerance: both are float32 sums of the same non-negative terms in different
orders, so they differ by at most (terms + a few roundings per term) 2^-24 of
their value: forward, up to 3 x 64 samples of 4 taps, 8e-5 at worst; back, up
to 700 lines a voxel, 1e-4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GRIDS = [(33, 20, 17), (20, 33, 16), (1, 24, 40), (24, 1, 31), (9, 7, 40), (16, 16, 1)]


def _lines(shape, count, rng):
    half = 0.5 * np.asarray(shape, dtype=np.float64)
    a = rng.normal(size=(count, 3))
    b = rng.normal(size=(count, 3))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    b /= np.linalg.norm(b, axis=1, keepdims=True)
    r = 1.4 * np.linalg.norm(half)
    p, q = a * r, b * r
    q[0::5] = -p[0::5] + rng.normal(size=p[0::5].shape)          # through the centre
    q[1::7] = 0.2 * q[1::7]                                        # end inside the image
    p[2::9, 1:], q[2::9, 1:] = 0.25, 0.25                          # along x, on the tap lattice or between
    p[3::9, [0, 2]], q[3::9, [0, 2]] = 0.0, 0.0                    # along y
    p[4::9, :2], q[4::9, :2] = 0.5, 0.5                            # along z
    q[5::11] = p[5::11] * [-1, -1, 1]                              # |dx| = |dy| for some
    p[5::11, 1], q[5::11, 1] = p[5::11, 0], q[5::11, 0]
    q[6::13] = p[6::13]                                            # no length
    p[7::13] *= 3.0
    q[7::13] = p[7::13] + [1.0, 0.5, 0.2]                          # outside
    return np.concatenate([p, q], axis=1).astype(np.float32)


@pytest.mark.parametrize("tof", [False, True])
@pytest.mark.parametrize("shape", GRIDS)
def test_quads_equal_image_walk(spect_lib, cuda, shape, tof):
    from paper_2309_01977_gb300 import pet
    rng = np.random.Generator(np.random.PCG64(sum(shape)))
    vox = int(np.prod(shape))
    short = max(1, vox // 32 - 1)  # lines of a call that walks the image
    n = max(700, vox // 32 + 1)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    lors = t(_lines(shape, n, rng))
    mult = t(rng.uniform(0.5, 1.5, size=n).astype(np.float32))
    q = t(rng.uniform(0.1, 1.0, size=n).astype(np.float32))
    bins = t(rng.integers(0, 7, size=n).astype(np.int32)) if tof else None
    x = t(rng.uniform(0.1, 2.0, size=shape).astype(np.float32))
    plan = pet.PetPlan(pet.PetGeometry(shape, (1.0, 1.0, 1.0), n_tof_bins=7, tof_bin_mm=6.0, tof_sigma_mm=4.0))
    cut = lambda v, s: None if v is None else v[s].contiguous()
    slices = [slice(k, k + short) for k in range(0, n, short)]
    fwd = plan.forward(x, lors, mult, tof_bin=bins)
    ref = torch.cat([plan.forward(x, cut(lors, s), cut(mult, s), tof_bin=cut(bins, s)) for s in slices])
    assert torch.all((fwd - ref).abs() <= 8e-5 * ref + 1e-30)
    assert float(ref.max()) > 0.0
    back = plan.back(q, lors, mult, tof_bin=bins)
    acc = torch.zeros(shape, device=cuda, dtype=torch.float64)
    for s in slices:
        acc += plan.back(cut(q, s), cut(lors, s), cut(mult, s), tof_bin=cut(bins, s)).double()
    assert torch.all((back.double() - acc).abs() <= 1e-4 * acc + 1e-30)
    plan.close()


# na mod 4 of 1, 2, 3, 0 along both walked axes, an odd and an even number of cells across
EM_GRIDS = [(5, 6, 9), (7, 8, 12), (2, 3, 33), (12, 21, 10)]


@pytest.mark.parametrize("tof", [False, True])
@pytest.mark.parametrize("shape", EM_GRIDS)
def test_quads_em_equals_its_parts(spect_lib, cuda, shape, tof):
    """An EM subiteration on quads is x back(1 / (forward(x) + s)) / sens of the two projectors above.  Both sum the
    same non-negative terms; the ratio is a few roundings: 2e-4 covers 700 lines a voxel twice over."""
    from paper_2309_01977_gb300 import pet
    rng = np.random.Generator(np.random.PCG64(sum(shape) + 1))
    n = 700
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    lors = t(_lines(shape, n, rng))
    mult = t(rng.uniform(0.5, 1.5, size=n).astype(np.float32))
    s = t(rng.uniform(0.1, 0.5, size=n).astype(np.float32))
    bins = t(rng.integers(0, 7, size=n).astype(np.int32)) if tof else None
    x = t(rng.uniform(0.1, 2.0, size=shape).astype(np.float32))
    sens = t(rng.uniform(0.5, 2.0, size=shape).astype(np.float32))
    plan = pet.PetPlan(pet.PetGeometry(shape, (1.0, 1.0, 1.0), n_tof_bins=7, tof_bin_mm=6.0, tof_sigma_mm=4.0))
    den = plan.forward(x, lors, mult, tof_bin=bins) + s
    ref = x * plan.back(1.0 / den, lors, mult, tof_bin=bins) / sens
    out = x.clone()
    plan.lm_osem(lors, mult, s, sens, out, 0, 1, tof_bin=bins)
    assert torch.all((out - ref).abs() <= 2e-4 * ref + 1e-30)
    assert float(ref.max()) > 0.0
    plan.close()


@pytest.mark.parametrize("radius", [1, 4, 8, 9, 14])
@pytest.mark.parametrize("shape", [(13, 17, 35), (8, 9, 32), (3, 2, 5)])
def test_blur_radii(spect_lib, cuda, shape, radius):
    """T_rr on both sides of the largest unrolled radius, wider and narrower than the axes: the back projection with
    it is the plain one blurred in float64 (2e-4: the two back projections' 1e-4, and 3 x 30 roundings)."""
    from paper_2309_01977_gb300 import pet
    rng = np.random.Generator(np.random.PCG64(sum(shape) + radius))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(cuda)
    lors = t(_lines(shape, 700, rng))
    q = t(rng.uniform(0.1, 1.0, size=700).astype(np.float32))
    sigma = radius / 3.0 - 0.05  # ceil(3 sigma) = radius
    plain = pet.PetPlan(pet.PetGeometry(shape, (1.0, 1.0, 1.0)))
    blurred = pet.PetPlan(pet.PetGeometry(shape, (1.0, 1.0, 1.0), rr_sigma_mm=sigma))
    ref = plain.back(q, lors).cpu().numpy().astype(np.float64)
    u = np.arange(-radius, radius + 1)
    w = np.exp(-u ** 2 / (2.0 * float(np.float32(sigma)) ** 2))
    w /= w.sum()
    for ax in range(3):
        ref = np.apply_along_axis(lambda v: np.convolve(v, w, mode="full")[radius:radius + len(v)], ax, ref)
    got = blurred.back(q, lors).cpu().numpy()
    assert np.all(np.abs(got - ref) <= 2e-4 * ref + 1e-30)
    plain.close()
    blurred.close()
