"""The quad walk in calls with as many lines as it is taken for, on the grids and
lines of test_gpu_pet_quads.py (700 lines of every kind), against the image walk
of short calls: a forward repeats the lines, a back projection and an OSEM
subiteration have them at random places among lines of weight 0, which add
nothing.  The launch counts show that quads were walked.

Tolerances as there: forward 8e-5, back 1e-4, an OSEM subiteration 2e-4.
"""
import numpy as np
import pytest

from test_gpu_pet_quads import EM_GRIDS, GRIDS, _lines

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LINES = {False: 50000, True: 530000}  # without and with time of flight


def _setup(shape, tof, seed):
    from paper_2309_01977_gb300 import pet
    rng = np.random.Generator(np.random.PCG64(seed))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    lors = t(_lines(shape, 700, rng))
    mult = t(rng.uniform(0.5, 1.5, size=700).astype(np.float32))
    bins = t(rng.integers(0, 7, size=700).astype(np.int32)) if tof else None
    x = t(rng.uniform(0.1, 2.0, size=shape).astype(np.float32))
    plan = pet.PetPlan(pet.PetGeometry(shape, (1.0, 1.0, 1.0), n_tof_bins=7, tof_bin_mm=6.0, tof_sigma_mm=4.0))
    # line of each place, and the places that carry weight (each line once)
    line = t(rng.integers(0, 700, size=LINES[tof]).astype(np.int64))
    place = t(rng.permutation(LINES[tof])[:700].astype(np.int64))
    line[place] = torch.arange(700, device="cuda")
    return rng, plan, lors, mult, bins, x, line, place


def _short(shape):
    """Slices of the 700 lines too short for quads."""
    step = max(1, int(np.prod(shape)) // 32 - 1)
    return [slice(k, min(700, k + step)) for k in range(0, 700, step)]


def _pick(v, s):
    return None if v is None else v[s].contiguous()


def _launches(spect_lib, fn):
    before = spect_lib.spect_kernel_launches()
    out = fn()
    return spect_lib.spect_kernel_launches() - before, out


def _forward(plan, shape, x, lors, mult, bins):
    return torch.cat([plan.forward(x, _pick(lors, s), _pick(mult, s), tof_bin=_pick(bins, s)) for s in _short(shape)])


def _back(plan, shape, q, lors, mult, bins):
    acc = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for s in _short(shape):
        acc += plan.back(_pick(q, s), _pick(lors, s), _pick(mult, s), tof_bin=_pick(bins, s)).double()
    return acc


@pytest.mark.parametrize("tof", [False, True])
@pytest.mark.parametrize("shape", GRIDS)
def test_projectors(spect_lib, cuda, shape, tof):
    rng, plan, lors, mult, bins, x, line, place = _setup(shape, tof, sum(shape))
    many = (_pick(lors, line), _pick(mult, line))
    n, got = _launches(spect_lib, lambda: plan.forward(x, *many, tof_bin=_pick(bins, line)))
    ref = _forward(plan, shape, x, lors, mult, bins)
    assert n == 5 and float(ref.max()) > 0.0
    assert torch.all((got - ref[line]).abs() <= 8e-5 * ref[line] + 1e-30)
    q = torch.from_numpy(rng.uniform(0.1, 1.0, size=700).astype(np.float32)).cuda()
    q_many = torch.zeros(line.numel(), device="cuda")
    q_many[place] = q
    n, got = _launches(spect_lib, lambda: plan.back(q_many, *many, tof_bin=_pick(bins, line)))
    ref = _back(plan, shape, q, lors, mult, bins)
    assert n == 5 and float(ref.max()) > 0.0
    assert torch.all((got.double() - ref).abs() <= 1e-4 * ref + 1e-30)
    plan.close()


@pytest.mark.parametrize("tof", [False, True])
@pytest.mark.parametrize("shape", EM_GRIDS)
def test_osem_subiteration(spect_lib, cuda, shape, tof):
    rng, plan, lors, mult, bins, x, line, place = _setup(shape, tof, sum(shape) + 1)
    s = torch.from_numpy(rng.uniform(0.1, 0.5, size=700).astype(np.float32)).cuda()
    sens = torch.from_numpy(rng.uniform(0.5, 2.0, size=shape).astype(np.float32)).cuda()
    den = _forward(plan, shape, x, lors, mult, bins) + s
    ref = x.double() * _back(plan, shape, 1.0 / den, lors, mult, bins) / sens.double()
    mult_many = torch.zeros(line.numel(), device="cuda")
    mult_many[place] = mult
    s_many, out = s[line].contiguous(), x.clone()
    n, _ = _launches(spect_lib, lambda: plan.lm_osem(_pick(lors, line), mult_many, s_many, sens, out, 0, 1,
                                                     tof_bin=_pick(bins, line)))
    assert n == 8 and float(ref.max()) > 0.0
    assert torch.all((out.double() - ref).abs() <= 2e-4 * ref + 1e-30)
    plan.close()
