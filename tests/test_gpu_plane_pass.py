"""The z+y pass over whole planes (needs a GPU): every length it takes on either axis, both directions,
in place, inside a convolution, and where the rule takes it."""

import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

Y_LENGTHS = [32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128]
Z_LENGTHS = [32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 125]


def _noise(shape, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)).astype(np.complex64)


def _takes(croft, shape):
    """Whether an AUTO plan's transforms and its convolutions run z and y as one pass."""
    with croft.Plan(*shape) as p:
        part = [s for s in p.describe().split(" | ") if "z+y in one pass" in s]
    return bool(part) and not part[0].startswith("convolutions: "), bool(part) and not part[0].startswith("transforms: ")


def _check_convolution(croft, shape):
    assert _takes(croft, shape)[1], shape
    x = _noise(shape, sum(shape))
    g = np.random.default_rng(6).uniform(0.1, 1, shape).astype(np.float32)
    d, dg = torch.from_numpy(x).cuda(), torch.from_numpy(g).cuda()
    with croft.Plan(*shape) as p, croft.Plan(*shape, schedule=croft.CROFT_SCHEDULE_THREE_PASS) as q:
        assert "fwd*G*bwd fused" in p.describe()
        y, z = p.convolve(d, dg), q.convolve(d, dg)
        p.convolve(d, dg, d)  # in place
        torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(z)), shape
    assert torch.equal(torch.view_as_real(y), torch.view_as_real(d)), shape
    assert oracle.rel_l2(y.cpu().numpy(), oracle.convolve(x, g)) <= 4e-6 * math.log2(x.size), shape


def _check(croft, shape):
    x = _noise(shape, sum(shape))
    tol = 2e-6 * math.log2(x.size)
    d = torch.from_numpy(x).cuda()
    assert _takes(croft, shape)[0], shape
    with croft.Plan(*shape) as p:
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
    if n <= 81:
        _check(croft_lib, (2, 32, n))
    elif n != 90:
        _check(croft_lib, (320, 36, n))
    if n <= 36:
        _check(croft_lib, (1, n, n))
    _check_convolution(croft_lib, (24 if n != 125 else 80, 32, n))


# one plane an SM and a rest; 256- and 128-thread CTAs; the largest planes the rule takes
@pytest.mark.parametrize("shape", [(150, 80, 54), (256, 80, 60), (300, 128, 36), (480, 96, 50), (480, 36, 125), (625, 36, 45),
                                   (480, 128, 32), (100, 36, 64)])
def test_many_planes(croft_lib, shape):
    _check(croft_lib, shape)


@pytest.mark.parametrize("shape", [(108, 54, 54), (160, 90, 45), (240, 45, 90), (320, 64, 75), (400, 40, 48), (640, 50, 60)])
def test_convolutions_of_many_planes(croft_lib, shape):
    _check_convolution(croft_lib, shape)


def test_rule(croft_lib):
    """(transforms, convolutions) of AUTO plans; other schedules run axis by axis."""
    for shape, takes in (((48, 48, 48), (True, True)), ((60, 60, 60), (False, False)), ((16, 64, 64), (False, False)),
                         ((80, 64, 64), (False, True)), ((120, 48, 48), (False, True)), ((120, 100, 32), (True, True)),
                         ((128, 60, 54), (True, False)), ((300, 48, 36), (True, True)), ((300, 64, 64), (False, False)),
                         ((300, 108, 108), (False, False)), ((8, 30, 32), (False, False)), ((8, 32, 256), (False, False)),
                         ((1, 36, 36), (True, False))):
        assert _takes(croft_lib, shape) == takes, shape
        with croft_lib.Plan(*shape, schedule=croft_lib.CROFT_SCHEDULE_THREE_PASS) as p:
            assert "z+y in one pass" not in p.describe(), shape
