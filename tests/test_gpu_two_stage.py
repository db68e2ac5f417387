"""The two-stage passes (needs a GPU): every length that has one, as row pass and as column pass over
short and long strides with ragged last tiles, against the oracle's axis DFT."""

import math
import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LENGTHS = [n for n in (2 ** a * 3 ** b * 5 ** c for a in range(11) for b in range(7) for c in range(5))
           if 32 < n <= 1024]


def _run(croft, shape, axis, direction, seed):
    rng = np.random.default_rng(seed)
    x = (rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)).astype(np.complex64)
    d = torch.from_numpy(x).cuda()
    out = torch.full_like(d, complex(float("nan"), 0))
    with croft.Plan(*shape) as p:
        desc = p.describe()
        croft.croft_exec_axes(p.handle, d, out, 1 << axis, direction)
        croft.croft_exec_axes(p.handle, d, d, 1 << axis, direction)  # in place
        torch.cuda.synchronize()
    y = out.cpu().numpy()
    assert np.array_equal(y.view(np.uint32), d.cpu().numpy().view(np.uint32))
    return x, y, [s for s in desc.split(" | ") if s.startswith("xyz"[axis] + ":")][0]


def _check(x, y, axis, direction):
    ref = oracle.dft_along_axis(x.astype(np.complex128), axis, direction)
    e = oracle.rel_l2(y, ref)
    assert e <= 2e-6 * math.log2(x.shape[axis]), (x.shape, axis, e)  # the bar of a transform of this length


@pytest.mark.parametrize("n", sorted(LENGTHS))
def test_every_length(croft_lib, n):
    # x: 75 columns; y: 27 columns in each of 2 planes; z: 15 rows (all ragged against the tiles)
    for shape, axis, direction in (((n, 3, 25), 0, -1), ((2, n, 27), 1, 1), ((5, 3, n), 2, -1)):
        x, y, desc = _run(croft_lib, shape, axis, direction, n + axis)
        if n not in (256, 972, 1000):
            assert "two-stage" in desc, desc
        _check(x, y, axis, direction)


@pytest.mark.parametrize("n", sorted(LENGTHS))
def test_every_length_with_the_general_kernels(croft_lib, monkeypatch, n):
    # (they run with CROFT_TWO_STAGE=0; the same ragged shapes)
    monkeypatch.setenv("CROFT_TWO_STAGE", "0")
    for shape, axis, direction in (((n, 3, 25), 0, 1), ((2, n, 27), 1, -1), ((5, 3, n), 2, 1)):
        x, y, desc = _run(croft_lib, shape, axis, direction, n + axis)
        assert "two-stage" not in desc, desc
        _check(x, y, axis, direction)


# the lengths whose kernels for long strides differ from those for short ones, and two whose do not
@pytest.mark.parametrize("n", [640, 675, 720, 729, 750, 768, 800, 810, 864, 1024])
def test_long_strides(croft_lib, n):
    # elements 262,440 bytes apart: the 16-column tile; 32,805 columns, five in the last tile
    x, y, desc = _run(croft_lib, (n, 81, 405), 0, -1, n)
    assert " W=16 " in desc.split("two-stage")[1], desc
    x, y = x.reshape(n, -1), y.reshape(n, -1)
    pick = np.r_[0:20, 16380:16390, x.shape[1] - 20:x.shape[1]]
    _check(x[:, pick], y[:, pick], 0, -1)


@pytest.mark.parametrize("n", [36, 108, 125, 256, 243, 360, 512, 625, 1024])
def test_convolution_with_ragged_tiles(croft_lib, n):
    # 135 columns of the fused axis (x; y of a 2D grid), the last tile partly filled
    for shape in ((n, 5, 27), (1, n, 135)):
        rng = np.random.default_rng(n)
        x = (rng.uniform(-1, 1, shape) + 1j * rng.uniform(-1, 1, shape)).astype(np.complex64)
        g = rng.uniform(0.1, 1, shape).astype(np.float32)
        with croft_lib.Plan(*shape) as p:
            assert "fwd*G*bwd fused" in p.describe()
            d = torch.from_numpy(x).cuda()
            y = p.convolve(d, torch.from_numpy(g).cuda())
            p.convolve(d, torch.from_numpy(g).cuda(), d)  # in place
            torch.cuda.synchronize()
        assert torch.equal(torch.view_as_real(y), torch.view_as_real(d))
        e = oracle.rel_l2(y.cpu().numpy(), oracle.convolve(x, g))
        assert e <= 4e-6 * math.log2(x.size), (shape, e)


@pytest.mark.parametrize("n", sorted(LENGTHS))
def test_no_less_precise_than_the_general_kernels(croft_lib, monkeypatch, n):
    """Rounding error against float64 over about four million points, as x and as z: other radices give 0.95 to 1.051 times the
    general kernels' error (a butterfly that rounds once more gave 1.06 and above at 54, 243, 288 and 324 points)."""
    rows = max(1, (1 << 22) // n)
    rows = max(k for k in (1024, 2048, 4096, 8192, 16384, 32768, 65536, 131072) if k <= rows)
    for axis, shape in ((0, (n, 64, rows // 64)), (2, (64, rows // 64, n))):
        gen = torch.Generator(device="cuda").manual_seed(n)
        x = torch.randn(shape, dtype=torch.complex64, device="cuda", generator=gen)
        ref = torch.fft.fft(x.to(torch.complex128), dim=axis)
        err = {}
        for two in ("0", "1"):
            monkeypatch.setenv("CROFT_TWO_STAGE", two)
            y = torch.empty_like(x)
            with croft_lib.Plan(*shape, schedule=croft_lib.CROFT_SCHEDULE_THREE_PASS) as p:
                croft_lib.croft_exec_axes(p.handle, x, y, 1 << axis, -1)
                torch.cuda.synchronize()
            err[two] = float((y - ref).norm() / ref.norm())
        assert err["1"] <= 1.058 * err["0"], (n, axis, err)


@pytest.mark.parametrize("switch,kernel,two", [(None, None, 3), ("CROFT_RING=0", None, 3), ("CROFT_PAIR=0", None, 3),
                                               ("CROFT_RING=1", "+ring", 2), ("CROFT_PAIR=1", "+pair", 2),
                                               ("CROFT_COL_TH=16", " T=16 ", 2), ("CROFT_TWO_STAGE=0", None, 0)])
def test_switches_name_their_own_kernels_only(croft_lib, monkeypatch, switch, kernel, two):
    """A measurement switch that names a kernel takes it for the passes it can serve (here x) and leaves the others
    alone; one that rules a kernel out leaves the two-stage kernels alone."""
    if switch:
        monkeypatch.setenv(*switch.split("="))
    with croft_lib.Plan(480, 36, 512) as p:
        d = p.describe()
    x = [s for s in d.split(" | ") if s.startswith("x:")][0]
    assert d.count("-> two-stage") == two, d
    assert ("-> two-stage" in x) == (kernel is None and two > 0), d
    assert kernel is None or kernel in x, d
    with croft_lib.Plan(48, 48, 48) as p:  # the plane pass has the two-stage passes' bits, and goes with them
        assert ("z+y in one pass" in p.describe()) == (two > 0), p.describe()


def test_slab_plans_build_each_table_once(croft_lib, monkeypatch):
    """The slab schedule of 1024^3 has over a thousand launches of the z and y axes; their tables are built once per axis
    (built per launch, creation took 17 times as long as with the general kernels)."""
    def create():
        best = math.inf
        for _ in range(5):
            t = time.perf_counter()
            with croft_lib.Plan(1024, 1024, 1024, schedule=croft_lib.CROFT_SCHEDULE_SLAB_L2):
                best = min(best, time.perf_counter() - t)
        return best

    two = create()
    monkeypatch.setenv("CROFT_TWO_STAGE", "0")
    general = create()
    assert two <= 4 * general, (two, general)
