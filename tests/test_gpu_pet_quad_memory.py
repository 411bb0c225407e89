"""The quads of the listmode PET walk are taken by the first call that needs
them: the image's by a forward, the back projection's by a back projection,
under stream capture and next to another thread's capture as well.  The launch
counts tell the walks apart: without T_rr a projector on quads is 5 kernels,
on the image 1; an EM subiteration 7 and 1, and its update.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SHAPE = (64, 64, 64)
SET = 16 * 64 * 65 * 65  # bytes of a set, at least


def _inputs(lines):
    rng = np.random.Generator(np.random.PCG64(5))
    a, b = rng.normal(size=(2, lines, 3))
    ends = [60.0 * v / np.linalg.norm(v, axis=1, keepdims=True) for v in (a, b)]
    lors = torch.from_numpy(np.concatenate(ends, axis=1).astype(np.float32)).cuda()
    x = torch.from_numpy(rng.uniform(0.1, 2.0, size=SHAPE).astype(np.float32)).cuda()
    q = torch.from_numpy(rng.uniform(0.1, 1.0, size=lines).astype(np.float32)).cuda()
    return x, lors, q


def _plan():
    from paper_2309_01977_gb300 import pet
    return pet.PetPlan(pet.PetGeometry(SHAPE, (1.0, 1.0, 1.0)))


def _launches(spect_lib, fn):
    before = spect_lib.spect_kernel_launches()
    fn()
    return spect_lib.spect_kernel_launches() - before


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


VOXELS = 64 ** 3


MANY = 3 << 14  # lines from which a back projection without time of flight walks quads


@pytest.mark.parametrize("lines,back", [(MANY, 5), (MANY - 1, 1), (VOXELS // 32, 1)])
def test_launches_tell_the_walks_apart(spect_lib, cuda, lines, back):
    x, lors, q = _inputs(lines)
    plan = _plan()
    one = torch.ones_like(x)
    assert _launches(spect_lib, lambda: plan.forward(x, lors)) == 5
    assert _launches(spect_lib, lambda: plan.back(q, lors)) == back
    assert _launches(spect_lib, lambda: plan.lm_osem(lors, q, None, one, x, 0, 1)) == 8
    few = VOXELS // 32 - 1
    lors, q = lors[:few].contiguous(), q[:few].contiguous()
    assert _launches(spect_lib, lambda: plan.forward(x, lors)) == 1
    assert _launches(spect_lib, lambda: plan.back(q, lors)) == 1
    assert _launches(spect_lib, lambda: plan.lm_osem(lors, q, None, one, x, 0, 1)) == 2
    plan.close()


@pytest.mark.parametrize("call", ["forward", "back"])
def test_a_projector_takes_its_own_set(spect_lib, cuda, call):
    x, lors, q = _inputs(MANY)
    warm = _plan()  # the kernels of both walks are loaded
    out = {"forward": torch.empty_like(q), "back": torch.empty_like(x)}
    run = lambda p: p.forward(x, lors, out=out[call]) if call == "forward" else p.back(q, lors, out=out[call])
    run(warm)
    plan = _plan()
    before = _free()
    run(plan)
    taken = before - _free()
    assert taken < 1.5 * SET, taken
    plan.close()
    warm.close()


def test_first_call_under_capture(spect_lib, cuda):
    x, lors, q = _inputs(VOXELS // 32)
    plan, ref = _plan(), _plan()
    want = ref.forward(x, lors)
    out = torch.zeros_like(q)
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        n = _launches(spect_lib, lambda: plan.forward(x, lors, out=out, stream=st))
    assert n == 5
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
    plan.close()
    ref.close()


def test_first_call_next_to_a_capture(spect_lib, cuda):
    """A plan's first call on one thread while another thread captures another stream."""
    x, lors, q = _inputs(VOXELS // 32)
    plan, ref = _plan(), _plan()
    want = ref.forward(x, lors)
    out = torch.zeros_like(q)
    side, st = torch.cuda.Stream(), torch.cuda.Stream()
    y = torch.zeros(1024, device=cuda)
    g = torch.cuda.CUDAGraph()
    counts = []
    torch.cuda.synchronize()

    def first_call():
        counts.append(_launches(spect_lib, lambda: plan.forward(x, lors, out=out, stream=side)))

    with torch.cuda.graph(g, stream=st):
        y.add_(1.0)
        t = threading.Thread(target=first_call)
        t.start()
        t.join()
    assert counts == [5]
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want) and float(y.min()) == 1.0
    assert _launches(spect_lib, lambda: plan.forward(x, lors, out=out, stream=side)) == 5
    plan.close()
    ref.close()
