"""Planes near the largest that shared memory holds, whose z tiles have an even
halo that is no multiple of 4: the forward stages their windows with 8-byte
loads.  Against the FP64 oracle at the parity bar of test_gpu_parity.py.
"""
import numpy as np
import pytest

from helpers import assert_close, f32, oracle_geom

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz", [(704, 48), (719, 20)])
def test_even_halo(spect_lib, oracle_mod, cuda, n, nz):
    slope = 5.1 / (n - 0.5)  # the nearest plane's radius is ceil(3 (0.5 + 5.1)) = 17
    g = spect_lib.Geometry(n=n, nz=nz, n_angles=1, angles_rad=[0.3], psf_slope=slope)
    rng = np.random.Generator(np.random.PCG64(n))
    f, mu = f32(rng.uniform(size=(n, n, nz))), f32(0.01 * rng.uniform(size=(n, n, nz)))
    og = oracle_geom(oracle_mod, g, mu)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(cuda)
    plan = spect_lib.Plan(g, t(mu))
    p_ref = oracle_mod.forward(f, og)
    assert_close(plan.forward(t(f)).cpu().numpy(), p_ref, 1e-5, "forward")
    plan.check()
    plan.close()
