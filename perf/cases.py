"""The transforms whose time is measured: what a program that uses this library has it do.

A case is one call of a plan that the program keeps: a forward or backward 3D transform, a PME
convolution, or a transform of a batch of grids.  Inputs and outputs are device tensors the
program owns; the output is written into a tensor kept beside the plan.

``op``: forward, backward or convolve on one (nx, ny, nz) grid; batch_forward or batch_backward on
the grids named in ``grids`` ("nx,ny,nz;nx,ny,nz;...").  ``dtype``: c64 (complex64, FP32
arithmetic), c128 (complex128), bf16x3 and fp16x3 (complex64 with a split-operand tensor-core
radix-16 stage).
"""

import math

import numpy as np
import torch

from paper_2002_04896_gb300 import croft

DTYPES = {"c64": croft.CROFT_C2C_F32, "c128": croft.CROFT_C2C_F64,
          "bf16x3": croft.CROFT_C2C_F32_TC_BF16X3, "fp16x3": croft.CROFT_C2C_F32_TC_FP16X3}

# axis lengths the library plans: 2^a 3^b 5^c up to 4096
LENGTHS = sorted(2 ** a * 3 ** b * 5 ** c for a in range(13) for b in range(8) for c in range(6)
                 if 2 <= 2 ** a * 3 ** b * 5 ** c <= 4096)
# complex128 lengths of useful size
LENGTHS_C128 = [32, 48, 60, 64, 96, 120, 128, 256]
# mesh axes of the per-system PME batch
BATCH_AXES = (48, 60, 64, 72, 80, 96, 120, 128)


def _grids_text(dims):
    return ";".join(",".join(str(int(v)) for v in d) for d in dims)


def _single(name, op, dtype, nx, ny, nz):
    c = {"op": op, "dtype": dtype, "nx": nx, "ny": ny, "nz": nz}
    return dict(c, name=name) if name else c


def _batch(name, op, dims):
    c = {"op": op, "dtype": "c64", "grids": _grids_text(dims)}
    return dict(c, name=name) if name else c


def listed():
    pme96 = np.random.default_rng(3).choice(np.asarray(BATCH_AXES), size=(96, 3))
    return [
        # the smallest grid in use: launch latency
        _single("forward_32", "forward", "c64", 32, 32, 32),
        # the reciprocal-space step of a small molecular system's PME mesh, every time step
        _single("convolve_108x108x80", "convolve", "c64", 108, 108, 80),
        # an ordinary mesh that fits in cache, the way back
        _single("backward_128", "backward", "c64", 128, 128, 128),
        # odd axis lengths, rows that do not fill their tiles
        _single("forward_225x243x200", "forward", "c64", 225, 243, 200),
        # the PME step of a mid-sized system
        _single("convolve_256", "convolve", "c64", 256, 256, 256),
        # a large mesh with three different mixed-radix axes
        _single("forward_384x360x320", "forward", "c64", 384, 360, 320),
        # a large cubic mixed-radix mesh, the way back
        _single("backward_480", "backward", "c64", 480, 480, 480),
        # the large power-of-two mesh
        _single("forward_512", "forward", "c64", 512, 512, 512),
        # the largest: a turbulence-sized field, axes longer than 512 points
        _single("forward_1024", "forward", "c64", 1024, 1024, 1024),
        # an ensemble of 96 small systems with meshes of different shapes in one call
        _batch("batch96_forward", "batch_forward", pme96),
        # double precision, for reference results
        _single("forward_128_c128", "forward", "c128", 128, 128, 128),
        # the tensor-core variant at the large mesh
        _single("forward_512_bf16x3", "forward", "bf16x3", 512, 512, 512),
    ]


def _near(lengths, v):
    return min(lengths, key=lambda n: abs(math.log(n / v)))


def _shape(rng, total, lengths):
    """Three lengths of about `total` points together, the axes within a factor of about two of each other."""
    side = total ** (1.0 / 3.0)
    a, b = math.exp(rng.uniform(-0.45, 0.45)), math.exp(rng.uniform(-0.45, 0.45))
    return _near(lengths, side * a), _near(lengths, side * b), _near(lengths, side / (a * b))


def draw(rng):
    kind = rng.choices(["c2c", "convolve", "plane", "batch", "c128", "tc"], weights=[40, 20, 8, 14, 9, 9])[0]
    way = rng.choice(["forward", "backward"])
    if kind in ("c2c", "convolve"):  # 32^3 to about 600^3 points
        total = math.exp(rng.uniform(math.log(2.0 ** 15), math.log(2.0 ** 27.5)))
        return _single(None, way if kind == "c2c" else "convolve", "c64", *_shape(rng, total, LENGTHS))
    if kind == "plane":  # one 2D field
        side = [_near(LENGTHS, math.exp(rng.uniform(math.log(256), math.log(4096)))) for _ in range(2)]
        return _single(None, way, "c64", 1, *side)
    if kind == "batch":  # ensembles of 6 to 128 systems
        count = round(math.exp(rng.uniform(math.log(6), math.log(128))))
        return _batch(None, "batch_" + way, [[rng.choice(BATCH_AXES) for _ in range(3)] for _ in range(count)])
    if kind == "c128":
        return _single(None, rng.choice(["forward", "backward", "convolve"]), "c128",
                       *(rng.choice(LENGTHS_C128) for _ in range(3)))
    tc_lengths = [n for n in LENGTHS if n % 16 == 0 and n <= 512]
    total = math.exp(rng.uniform(math.log(2.0 ** 18), math.log(2.0 ** 27)))
    return _single(None, way, rng.choice(["bf16x3", "fp16x3"]), *_shape(rng, total, tc_lengths))


def _dims(case):
    if "grids" in case:
        return [tuple(int(v) for v in d.split(",")) for d in case["grids"].split(";")]
    return [(case["nx"], case["ny"], case["nz"])]


def _complex(case):
    return torch.complex128 if case["dtype"] == "c128" else torch.complex64


def _charges(shape, gen, dtype):
    """A PME charge mesh: +-1 charges, one per 16 mesh points and at most 8 million, at random
    positions, spread with order-4 B-splines; imaginary part zero.  Accumulated in fixed point, so
    that the same seed gives the same bits."""
    total = math.prod(shape)
    n = max(2, min(8_000_000, total // 16))
    n -= n % 2
    q = torch.ones(n, dtype=torch.float64, device="cuda")
    q[::2] = -1.0
    idx, wts = [], []
    for length in shape:
        u = torch.rand(n, generator=gen, dtype=torch.float64, device="cuda") * length
        i0 = u.floor()
        w = u - i0
        wts.append([(1 - w) ** 3 / 6, (3 * w ** 3 - 6 * w ** 2 + 4) / 6, (-3 * w ** 3 + 3 * w ** 2 + 3 * w + 1) / 6,
                    w ** 3 / 6])
        idx.append([(i0.long() + t) % length for t in (-1, 0, 1, 2)])
    mesh = torch.zeros(total, dtype=torch.int64, device="cuda")
    for i in range(4):
        for j in range(4):
            row = (idx[0][i] * shape[1] + idx[1][j]) * shape[2]
            wij = q * wts[0][i] * wts[1][j] * 2.0 ** 40
            for k in range(4):
                mesh.index_add_(0, row + idx[2][k], (wij * wts[2][k]).round().long())
    out = torch.zeros(shape, dtype=dtype, device="cuda")
    out.real.copy_((mesh.double() * 2.0 ** -40).view(shape))
    return out


def _field(shape, gen, dtype):
    """A complex Gaussian field (a turbulence snapshot, or a spectrum on its way back)."""
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    x = torch.randn(tuple(shape) + (2,), generator=gen, dtype=real, device="cuda")
    return torch.view_as_complex(x)


def _input(case, seed):
    """The input grids of a case, and the influence function of a convolution (else None)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    dims, dtype = _dims(case), _complex(case)
    pme = case["op"] in ("convolve", "batch_forward") or (case["op"] == "forward" and dims[0][0] != 1
                                                          and math.prod(dims[0]) <= 2 ** 28)
    grids = [(_charges if pme else _field)(d, gen, dtype) for d in dims]
    if case["op"] != "convolve":
        return grids, None
    # The smooth-PME influence function on a box of spacing 0.1 with Ewald parameter 3.12 (the
    # interpolation's correction left at its small-wavenumber form).
    f2 = torch.zeros(dims[0], dtype=torch.float64, device="cuda")
    for a, length in enumerate(dims[0]):
        k = torch.fft.fftfreq(length, d=0.1, dtype=torch.float64, device="cuda")
        f2 += (k * k).view([-1 if b == a else 1 for b in range(3)])
    f2[0, 0, 0] = 1.0
    g = torch.exp(-(math.pi / 3.12) ** 2 * f2) / (math.pi * math.prod(dims[0]) * 1e-3 * f2)
    g[0, 0, 0] = 0.0
    return grids, g.to(torch.float64 if dtype == torch.complex128 else torch.float32)


def prepare(case, seed):
    grids, g = _input(case, seed)
    dims = _dims(case)
    if case["op"].startswith("batch_"):
        # one allocation for the whole ensemble's results, every grid 256-byte aligned
        starts, end = [], 0
        for d in dims:
            starts.append(end)
            end += -(-math.prod(d) // 32) * 32
        flat = torch.zeros(end, dtype=torch.complex64, device="cuda")
        outs = [flat[s:s + math.prod(d)].view(d) for s, d in zip(starts, dims)]
        plan = croft.BatchPlan(dims, mode=croft.CROFT_BATCH_GROUPED)
        return {"op": case["op"], "plan": plan, "ins": grids, "outs": outs, "flat": flat}
    plan = croft.Plan(*dims[0], dtype=DTYPES[case["dtype"]])
    return {"op": case["op"], "plan": plan, "x": grids[0], "g": g, "y": torch.empty_like(grids[0])}


def run(state):
    op, plan = state["op"], state["plan"]
    if op == "forward":
        return plan.forward(state["x"], state["y"])
    if op == "backward":
        return plan.backward(state["x"], state["y"])
    if op == "convolve":
        return plan.convolve(state["x"], state["g"], state["y"])
    if op == "batch_forward":
        plan.forward(state["ins"], state["outs"])
    else:
        plan.backward(state["ins"], state["outs"])
    return state["flat"]


def work(case):
    """Each grid read once and written once (a convolution reads the influence function too);
    5 N log2 N operations per transform."""
    element = 16 if case["dtype"] == "c128" else 8
    nbytes = flops = 0
    for d in _dims(case):
        n = math.prod(d)
        nbytes += 2 * element * n
        flops += 5 * n * math.log2(max(2, n))
    if case["op"] == "convolve":
        nbytes += element // 2 * math.prod(_dims(case)[0])
        flops *= 2
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error against 64 bits of a transform: measured 1.3e-7 to 2.0e-7 for complex64
    (2.1e-7 for a convolution), 4.3e-16 to 4.9e-16 for complex128, 5.4e-6 for bf16x3."""
    rel = {"c64": 8e-7, "c128": 2e-15, "bf16x3": 2.2e-5, "fp16x3": 3e-6}[case["dtype"]]
    return {"rel": 1.25 * rel if case["op"] == "convolve" else rel}


def exact(case, seed):
    grids, g = _input(case, seed)
    dims = _dims(case)
    if case["op"] == "convolve":
        y = torch.fft.fftn(grids[0].to(torch.complex128))
        y *= g.double()
        return torch.fft.ifftn(y, norm="forward")
    if case["op"] == "forward":
        return torch.fft.fftn(grids[0].to(torch.complex128))
    if case["op"] == "backward":
        return torch.fft.ifftn(grids[0].to(torch.complex128), norm="forward")
    flat = []
    for d, x in zip(dims, grids):
        x = x.to(torch.complex128)
        y = torch.fft.fftn(x) if case["op"] == "batch_forward" else torch.fft.ifftn(x, norm="forward")
        flat.append(y.reshape(-1))
        flat.append(torch.zeros(-math.prod(d) % 32, dtype=torch.complex128, device="cuda"))
    return torch.cat(flat)
