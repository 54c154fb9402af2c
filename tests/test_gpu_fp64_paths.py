"""Paths that few right-hand sides take against the general ones on the same
plan: the symmetric FP64 translations (up to 4 columns) against near_kernel
(9 columns), and the row-per-lane up/down passes (up to 8 columns, 4 in
complex128) against the column-per-lane ones.

The same sums in another order: FP64 within 1e-13 of max |u| (sums of ~10^4
terms), FP32 within 4e-6 (each side within 2e-6 of FP64)."""
import math

import numpy as np
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


CASES = [("laplace3d", 1, 8), ("laplace3d", 33, 64), ("laplace3d", 700, 24), ("laplace3d", 6000, 128),
         ("laplace2d", 65, 64), ("laplace2d", 5000, 31), ("helmholtz3d", 900, 40), ("helmholtz2d", 2500, 64)]


@pytest.mark.parametrize("kind,n,leaf", CASES)
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32", 4e-6)])
def test_few_columns_match_many(kind, n, leaf, precision, tol):
    dim = 2 if kind.endswith("2d") else 3
    x = W.points_uniform(n, dim, 81) if n < 64 else clustered(n, dim, 81)
    if n > 100:
        x[7] = x[3]                                            # coincident points contribute nothing
    f = SkelFMM(x, kind, 1e-8, leaf, nrhs_max=9, kappa=20.0 if kind.startswith("helm") else 0.0)
    cplx = kind.startswith("helm")
    q = (W.charges_complex if cplx else W.charges_normal)(x.shape[0], 9, 82)
    q = torch.from_numpy(np.ascontiguousarray(q)).cuda()
    if precision == "fp32":
        q = q.to(torch.complex64 if cplx else torch.float32)
    for fn in (f.apply, f.apply_transpose):
        ref = fn(q, precision)
        scale = max(float(ref.abs().max()), 1e-30)
        for m in (1, 2, 3, 4, 5, 8):
            got = fn(q[:, :m].contiguous(), precision)
            assert float((got - ref[:, :m]).abs().max()) <= tol * scale, m
            assert torch.equal(fn(q[:, :m].contiguous(), precision), got)


def test_log_of_distances_over_many_scales():
    """2D Laplace of pairs from 1e-150 to 1e150 apart (r^2 normal, and beyond
    the table's range): each potential of a two-point set is -log r / 2 pi."""
    for r in [1e-150, 3e-20, 1e-8, 0.5, 0.7071, 0.99999999, 1.0, 1.0000001, 1.4142, 2.0, 7.3, 1e5, 1e150]:
        f = SkelFMM(np.array([[0.0, 0.0], [r, 0.0]]), "laplace2d", 1e-8, 4, nrhs_max=1)
        u = f.apply(torch.tensor([0.0, 1.0], dtype=torch.float64, device="cuda"), "fp64")
        want = -math.log(r) / (2 * math.pi)
        assert abs(float(u[0]) - want) <= 4e-16 * abs(want) + 1e-17, r
        assert float(u[1]) == 0.0
