"""A new attenuation map on a kept plan gives the sensitivities of a fresh plan, bit for bit.

With a field-of-view mask the first kernel after the one that writes the
attenuation cache is the FP32 back blur, which copies its first plane of the
cache ahead of the wait of an early launch: that launch has to be an ordinary
one.  Maps alternate, so that a plane left from the map before shows.
"""
import numpy as np
import pytest

from helpers import phantom_inputs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nz,psf_bf16", [(40, 36, False), (64, 64, False), (132, 44, False), (64, 64, True)])
def test_set_mu_on_masked_plan(n, nz, psf_bf16):
    from paper_2309_01977_gb300 import spect
    fov = np.ones((8, n, nz), dtype=np.float32)
    fov[:, :2] = 0.25
    fov[:, :, :1] = 0.5
    g = spect.Geometry(n=n, nz=nz, n_angles=8, n_subsets=2, psf_bf16=psf_bf16, fov_mask=fov)
    mus = [torch.from_numpy(phantom_inputs(n, nz, seed)[1].astype(np.float32)).cuda() for seed in (3, 4)]
    mus[1] = 3.0 * mus[1] + 0.02
    want = []
    for mu in mus:
        fresh = spect.Plan(g, mu)
        want.append([fresh.sensitivity(m).clone() for m in range(2)])
        fresh.close()
    assert not torch.equal(want[0][0], want[1][0])
    kept = spect.Plan(g, mus[0])
    for turn in range(6):
        which = (turn + 1) % 2
        spect.spect_plan_set_mu(kept.handle, mus[which])
        for m in range(2):
            assert torch.equal(kept.sensitivity(m), want[which][m]), (turn, m)
    kept.close()
