"""The on-the-fly tensor-core kernel at the edges of its work division: lists
shorter than a pair of tiles, whole and ragged segments, items that share a
CTA, lists cut over several CTAs (small plans), and right-hand sides that end
inside a pass. Every column against the FP64 apply of the same plan within
2e-6 of max |u|, the bound the tensor-core path is held to elsewhere (3-pass
TF32 split, FP32 sums: measured 3e-7)."""
import pytest
import torch

from paper_2310_16668_gb300 import SkelFMM
from paper_2310_16668_gb300 import workloads as W
from tests._util import clustered

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_16668_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("kind,n,leaf,dist", [
    ("laplace3d", 5, 8, "uniform"),            # one leaf, one short tile
    ("laplace3d", 300, 300, "uniform"),        # one leaf of two full items and a ragged one
    ("laplace3d", 4500, 4500, "uniform"),      # lists of 141 tiles, pairs of items, cut into segments
    ("laplace3d", 9001, 64, "uniform"),
    ("laplace3d", 7000, 24, "clustered"),
    ("laplace2d", 6000, 33, "clustered"),
    ("laplace3d", 90000, 128, "uniform"),      # whole lists
])
@pytest.mark.parametrize("nrhs", [4, 45])
def test_units_match_fp64(kind, n, leaf, dist, nrhs):
    dim = 2 if kind.endswith("2d") else 3
    x = W.points_uniform(n, dim, 71) if dist == "uniform" else clustered(n, dim, 71)
    f = SkelFMM(x, kind, 1e-6, leaf, nrhs_max=nrhs)
    q = torch.from_numpy(W.charges_normal(x.shape[0], nrhs, 72)).cuda().float()
    u = f.apply(q, "fp32_tc")
    f.device_status()
    ref = f.apply(q.double(), "fp64")
    err = (u.double() - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(err.max()) < 2e-6
    assert torch.equal(f.apply(q, "fp32_tc"), u)


def test_log_of_small_distances():
    """2D, distances of 1e-20 to 1e-17 (r^2 from subnormal to normal FP32, and 0
    for coincident points). Unit charges, so that a column is single kernel
    values: r^2 = 1e-40 has a rounding error of 1e-5, 1e-7 of its logarithm, the
    logarithm rounds to 1e-7 and the 3-pass split to 5e-7."""
    n = 700
    x = W.points_uniform(n, 2, 73) * 1e-17
    x[1::7] = x[::7] + 1e-20
    x[2::7] = x[::7]
    f = SkelFMM(x, "laplace2d", 1e-6, n, nrhs_max=33)
    q = torch.zeros((n, 33), device="cuda")
    q[torch.arange(33) * 21, torch.arange(33)] = 1.0
    u = f.apply(q, "fp32_tc")
    ref = f.apply(q.double(), "fp64")
    f.device_status()
    err = (u.double() - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(err.max()) < 2e-6
