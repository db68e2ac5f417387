"""Half tiles of the complex128 passes (``croft_half_tiles64`` in ``csrc/croft_sched.h``) at the edges of
the tiles, against the FP64 oracle (needs a GPU).

Tolerance: relative L2 <= 1e-14 * log2(N) (double-precision rounding of an O(log N)-deep transform).
"""

import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# half tiles in all three passes; tiles that end inside a half; one pencil; lengths without a narrower tile; half tiles in one
# axis only; several rounds of tiles
@pytest.mark.parametrize("shape", [(16, 16, 16), (15, 10, 6), (5, 128, 3), (256, 3, 3), (512, 5, 2), (64, 1, 64),
                                   (60, 96, 120), (256, 64, 64), (2, 1, 1), (1024, 15, 1)])
def test_f64_tiles(croft_lib, shape):
    r = np.random.default_rng(sum(shape))
    x = r.uniform(-1, 1, shape) + 1j * r.uniform(-1, 1, shape)
    tol = 1e-14 * max(1.0, math.log2(x.size))
    d = torch.from_numpy(x).cuda()
    with croft_lib.Plan(*shape, dtype=croft_lib.CROFT_C2C_F64) as p:
        yf, yb = p.forward(d), p.backward(d)
        z = p.backward(yf, yf)  # in place
        torch.cuda.synchronize()
    assert oracle.rel_l2(yb.cpu().numpy(), oracle.backward(x)) <= tol
    assert oracle.rel_l2(z.cpu().numpy(), x.size * x) <= tol
    with croft_lib.Plan(*shape, dtype=croft_lib.CROFT_C2C_F64) as p:
        assert oracle.rel_l2(p.forward(d).cpu().numpy(), oracle.forward(x)) <= tol
