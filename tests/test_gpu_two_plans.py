"""Plans that share a kernel, alive at once (needs a GPU): a kernel's limit on dynamic shared memory
belongs to the function, so a plan whose tiles need less must leave it where an older plan needs it.

Tolerance: relative L2 <= 2e-6 * log2(N) against the FP64 oracle.
"""

import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _input(shape, seed, dtype=np.complex64):
    r = np.random.default_rng(seed)
    return (r.uniform(-1, 1, shape) + 1j * r.uniform(-1, 1, shape)).astype(dtype)


# (older plan, newer plan): planes of the same y length, the newer ones smaller in shared memory; below and above 48 KB
@pytest.mark.parametrize("older,newer", [((64, 36, 64), (64, 36, 32)), ((8, 128, 32), (256, 128, 36))])
def test_plane_pass_plans(croft_lib, older, newer):
    with croft_lib.Plan(*older) as a, croft_lib.Plan(*newer) as b:
        for plan, shape in ((a, older), (b, newer), (a, older)):
            assert "z+y in one pass" in plan.describe(), shape
            x = _input(shape, sum(shape))
            d = torch.from_numpy(x).cuda()
            g = torch.ones(shape, dtype=torch.float32, device="cuda")
            y, z, c = plan.forward(d), plan.backward(d), plan.convolve(d, g)
            torch.cuda.synchronize()
            tol = 2e-6 * math.log2(x.size)
            assert oracle.rel_l2(y.cpu().numpy(), oracle.forward(x)) <= tol, shape
            assert oracle.rel_l2(z.cpu().numpy(), oracle.backward(x)) <= tol, shape
            assert oracle.rel_l2(c.cpu().numpy(), x.size * x.astype(np.complex128)) <= 2 * tol, shape


# complex128 rows of 1024 points: full tiles of the older plan, half tiles of the newer one
def test_complex128_row_plans(croft_lib):
    older, newer = (64, 64, 1024), (96, 64, 1024)
    f64 = croft_lib.CROFT_C2C_F64
    with croft_lib.Plan(*older, dtype=f64) as a, croft_lib.Plan(*newer, dtype=f64) as b:
        for plan, shape in ((a, older), (b, newer), (a, older)):
            x = torch.from_numpy(_input(shape, 7, np.complex128)).cuda()
            y = torch.empty_like(x)
            croft_lib.croft_exec_axes(plan.handle, x, y, 4, -1)  # the z axis
            torch.cuda.synchronize()
            e = oracle.rel_l2(y[::16].cpu().numpy(), oracle.dft_along_axis(x[::16].cpu().numpy(), 2, -1))
            assert e <= 1e-14 * math.log2(1024), (shape, e)
