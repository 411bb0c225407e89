"""FP32 sensitivities are the back projection of all-ones data, bit for bit: the
sums over the taps that their kernel forms per distance from the plane's edges
have the order and the roundings of the back blur.  Planes wider and narrower
than the PSF along y and z, one z tile and several, per-angle PSF tables, one
group of angles and several, with and without attenuation and PSF.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

CASES = {
    "64": dict(n=64, nz=64, n_angles=12, n_subsets=3),
    "tiny": dict(n=3, nz=4, n_angles=4, n_subsets=2, psf_sigma0=2.0),
    "narrow_y": dict(n=24, nz=60, n_angles=6, n_subsets=2, psf_sigma0=4.0),   # 2 R + 1 > n
    "narrow_z": dict(n=64, nz=8, n_angles=6, n_subsets=2, psf_sigma0=3.0),    # 2 R + 1 > nz
    "tiles": dict(n=100, nz=180, n_angles=4, n_subsets=2, psf_slope=0.05),
    "orbit": dict(n=48, nz=40, n_angles=6, n_subsets=2, det_offsets=[1.0 + 2.0 * a for a in range(6)]),
    "groups": dict(n=33, nz=24, n_angles=40, n_subsets=2),                    # 20 angles: 16 and 4
    "bare": dict(n=40, nz=36, n_angles=6, n_subsets=2, attenuation=False),
    "no_psf": dict(n=40, nz=36, n_angles=6, n_subsets=2, psf=False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_sensitivity_is_the_back_projection_of_ones(spect_lib, cuda, name):
    kw = CASES[name]
    g = spect_lib.Geometry(**kw)
    mu = None
    if kw.get("attenuation", True):
        rng = np.random.Generator(np.random.PCG64(kw["n"]))
        mu = torch.from_numpy(rng.uniform(0.0, 0.1, size=(g.n, g.n, g.nz)).astype(np.float32)).to(cuda)
    plan = spect_lib.Plan(g, mu)
    for m in range(g.n_subsets):
        ones = torch.ones((g.n_angles // g.n_subsets, g.n, g.nz), device=cuda)
        sens = plan.sensitivity(m)
        assert float(sens.max()) > 0.0
        assert torch.equal(sens, plan.back(ones, subset=m)), m
    plan.check()
    plan.close()
