"""Forward and back projection where the FP32 plane kernels change shape:
one z tile and several, a last tile narrower than the others, CTAs of 256
and 512 threads, radii on both sides of the narrow variants' largest (14),
the largest radius (20) and none, odd and tiny planes, and no attenuation.
Against the FP64 oracle at the parity bar of test_gpu_parity.py.
"""
import numpy as np
import pytest

from helpers import assert_close, f32, oracle_geom, phantom_inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1e-5

CASES = {
    "smallest": dict(n=2, nz=4, n_angles=3),
    "odd33x24": dict(n=33, nz=24, n_angles=5),
    "strip_edge48x64": dict(n=48, nz=64, n_angles=4),
    "strip_past49x68": dict(n=49, nz=68, n_angles=4),
    "r14_52x40": dict(n=52, nz=40, n_angles=4, psf_sigma0=1.5, psf_slope=0.06),
    "r15_52x40": dict(n=52, nz=40, n_angles=4, psf_sigma0=1.8, psf_slope=0.06),
    "two_tiles160x148": dict(n=160, nz=148, n_angles=2),
    "narrow_last_tile148x180": dict(n=148, nz=180, n_angles=2, psf_slope=0.02),
    "r20_tiles120x160": dict(n=120, nz=160, n_angles=2, psf_slope=0.05),
    "tall32x300": dict(n=32, nz=300, n_angles=3),
    "bare_tiles144x136": dict(n=144, nz=136, n_angles=2, attenuation=False),
    "no_psf_tiles150x200": dict(n=150, nz=200, n_angles=2, psf=False),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_plane_shapes(spect_lib, oracle_mod, cuda, name):
    g = spect_lib.Geometry(**CASES[name])
    rng = np.random.Generator(np.random.PCG64(77))
    if g.n >= 32:
        f, mu = phantom_inputs(g.n, g.nz, 31)
        f = f32(f + 0.05 * rng.uniform(size=f.shape))  # nonzero up to the edges
    else:
        f, mu = f32(rng.uniform(size=(g.n, g.n, g.nz))), f32(0.2 * rng.uniform(size=(g.n, g.n, g.nz)))
    og = oracle_geom(oracle_mod, g, mu)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(cuda)
    plan = spect_lib.Plan(g, t(mu) if g.attenuation else None)
    p_ref = oracle_mod.forward(f, og)
    assert_close(plan.forward(t(f)).cpu().numpy(), p_ref, TOL, (name, "forward"))
    q = f32(rng.uniform(0.0, 2.0, size=p_ref.shape))
    assert_close(plan.back(t(q)).cpu().numpy(), oracle_mod.back(q, og), TOL, (name, "back"))
    plan.check()
    plan.close()
