"""The z+y pass over whole planes (needs a GPU): every length it takes on either axis, both directions,
in place, inside a convolution, and where the rule takes it."""

import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

Y_LENGTHS = [32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128]
Z_LENGTHS = [32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 81, 125]


def _noise(shape, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)).astype(np.complex64)


def _check(croft, shape):
    x = _noise(shape, sum(shape))
    tol = 2e-6 * math.log2(x.size)
    d = torch.from_numpy(x).cuda()
    with croft.Plan(*shape) as p:
        assert "z+y in one pass" in p.describe(), p.describe()
        assert croft.croft_plan_num_launches(p.handle) == (2 if shape[0] > 1 else 1)
        out = torch.full_like(d, complex(float("nan"), 0))
        p.forward(d, out)
        b = p.backward(d)
        c = d.clone()
        p.forward(c, c)
        torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(c))
        croft.croft_plan_set_timing(p.handle, True)  # an axis at a time
        t = p.forward(d)
        u = p.backward(d)
        n = len(croft.croft_plan_pass_times(p.handle))
        assert n == croft.croft_plan_num_launches(p.handle) == (3 if shape[0] > 1 else 2)
        croft.croft_plan_set_timing(p.handle, False)
        a = torch.empty_like(d)
        croft.croft_exec_axes(p.handle, d, a, 7, -1)
    with croft.BatchPlan([shape], mode=croft.CROFT_BATCH_GROUPED) as p:
        (g,) = p.forward([d])
        torch.cuda.synchronize()
    # the passes' own splits and sums: the same bits axis by axis, timed, and in a batch
    for other in (t, a, g):
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(other)), shape
    assert torch.equal(torch.view_as_real(b), torch.view_as_real(u)), shape
    assert oracle.rel_l2(out.cpu().numpy(), oracle.forward(x)) <= tol, shape
    assert oracle.rel_l2(b.cpu().numpy(), oracle.backward(x)) <= tol, shape


@pytest.mark.parametrize("n", Y_LENGTHS)
def test_every_length_as_y(croft_lib, n):
    _check(croft_lib, (3, n, 32))


@pytest.mark.parametrize("n", Z_LENGTHS)
def test_every_length_as_z(croft_lib, n):
    _check(croft_lib, (2, 32, n) if n <= 72 else (400, 36, n))
    if n <= 36:
        _check(croft_lib, (1, n, n))


# one plane an SM and a rest; 256- and 128-thread CTAs; the largest planes the rule takes
@pytest.mark.parametrize("shape", [(150, 100, 45), (256, 80, 60), (300, 128, 36), (480, 96, 50), (480, 36, 125), (625, 36, 45),
                                   (480, 128, 32), (100, 36, 64)])
def test_many_planes(croft_lib, shape):
    _check(croft_lib, shape)


def test_convolution_and_rule(croft_lib):
    shape = (20, 48, 45)
    x = _noise(shape, 5)
    g = np.random.default_rng(6).uniform(0.1, 1, shape).astype(np.float32)
    with croft_lib.Plan(*shape) as p:
        assert "z+y in one pass" in p.describe() and "fwd*G*bwd fused" in p.describe()
        y = p.convolve(torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda())
        torch.cuda.synchronize()
    assert oracle.rel_l2(y.cpu().numpy(), oracle.convolve(x, g)) <= 4e-6 * math.log2(x.size)
    for shape, takes in (((48, 48, 48), True), ((60, 60, 60), False), ((16, 64, 64), False), ((120, 48, 48), False),
                         ((120, 100, 32), True), ((128, 60, 54), True), ((300, 48, 36), True), ((300, 64, 64), False),
                         ((300, 108, 108), False), ((8, 30, 32), False), ((8, 32, 256), False)):
        with croft_lib.Plan(*shape) as p:
            assert ("z+y in one pass" in p.describe()) == takes, shape
        with croft_lib.Plan(*shape, schedule=croft_lib.CROFT_SCHEDULE_THREE_PASS) as p:
            assert "z+y in one pass" not in p.describe(), shape
