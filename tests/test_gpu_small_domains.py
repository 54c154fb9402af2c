"""2D Laplace on the tensor cores where squared distances are subnormal FP32
numbers between boxes that do not touch: a square of side 3e-19, leaves of 64
(its finest boxes are 1.9e-20 wide, so r^2 there starts at 3.5e-40).

Bound, per target: 2e-6 of max |u| (what the tensor-core path is held to
elsewhere), and the rounding of r^2: squares and their sum round to multiples of
2^-149, two half units, so a kernel value -log(r^2) / 4 pi is off by 2^-149 / r^2
/ 4 pi. Points on a jittered grid (no pair closer than a fifth of its spacing)
and charges between 0.5 and 1.5: nothing cancels."""
import math

import numpy as np
import pytest
import torch

from paper_2310_16668_gb300 import SkelBatch, SkelFMM
from paper_2310_16668_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIDE = 3e-19


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_16668_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _points():
    g = (np.arange(55) + 0.5) / 55
    x = np.stack(np.meshgrid(g, g), -1).reshape(-1, 2)
    return SIDE * (x + np.random.default_rng(91).uniform(-0.4, 0.4, x.shape) / 55)


def _rounding(x):
    """max over targets of the sum of 1.5 * 2^-149 / r^2 / 4 pi."""
    worst = 0.0
    for p in x:
        r2 = ((x - p) ** 2).sum(1)
        worst = max(worst, float((1.5 * 2.0 ** -149 / r2[r2 > 0]).sum()))
    return worst / (4 * math.pi)


@pytest.mark.parametrize("form", ["on the fly", "stored", "symmetric", "merged"])
@pytest.mark.parametrize("nrhs", [4, 33])
def test_subnormal_distances_between_far_boxes(form, nrhs):
    x = _points()
    n = x.shape[0]
    lo = 0
    if form == "merged":                       # with a set of ordinary size before it
        b = SkelBatch([W.points_uniform(700, 2, 92), x], "laplace2d", 1e-6, 64, nrhs_max=nrhs)
        f = b.merged()
        lo = 700
    else:
        f = SkelFMM(x, "laplace2d", 1e-6, 64, nrhs_max=nrhs, store_tiles={"stored": 1, "symmetric": 2}.get(form, 0))
    q = torch.from_numpy(np.random.default_rng(93).uniform(0.5, 1.5, (lo + n, nrhs))).cuda().float()
    if lo:
        u, ref = torch.empty((nrhs, lo + n), device="cuda"), torch.empty((nrhs, lo + n), device="cuda", dtype=torch.float64)
        f.apply_into(q.t().contiguous(), u, nrhs, "fp32_tc")
        f.apply_into(q.double().t().contiguous(), ref, nrhs, "fp64")
        u, ref = u.t()[lo:], ref.t()[lo:]
    else:
        u, ref = f.apply(q, "fp32_tc"), f.apply(q.double(), "fp64")
    f.device_status()
    scale = float(ref.abs().max())
    err = float((u.double() - ref).abs().max())
    assert err <= 2e-6 * scale + _rounding(x), (err, scale)
