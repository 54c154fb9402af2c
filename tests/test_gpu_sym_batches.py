"""The symmetric FP64 translations in batches that share one buffer of slots:
plans with more slots than a batch holds (2^21), against near_kernel (9
columns), and the memory a plan spends on them.

FP64 within 1e-13 of max |u| (the same sums of ~10^4 terms in another order)."""
import numpy as np
import pytest
import torch

from paper_2310_16668_gb300 import SkelFMM
from paper_2310_16668_gb300 import workloads as W
from tests._util import clustered

pytestmark = pytest.mark.gpu

BATCH = 1 << 21                                # slots of a batch, 32 rows of FP64 per column each


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_16668_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("kind,n,dist", [("laplace3d", 262144, "uniform"), ("laplace3d", 300000, "clustered"),
                                         ("helmholtz3d", 200000, "uniform")])
def test_batches_match_general_translations(kind, n, dist):
    x = W.points_uniform(n, 3, 95) if dist == "uniform" else clustered(n, 3, 95)
    cplx = kind.startswith("helm")
    f = SkelFMM(x, kind, 1e-6, 128, nrhs_max=9, kappa=10.0 if cplx else 0.0, device_build=True)
    q = (W.charges_complex if cplx else W.charges_normal)(x.shape[0], 9, 96)
    q = torch.from_numpy(np.ascontiguousarray(q)).cuda()
    ref = f.apply(q, "fp64")
    scale = float(ref.abs().max())
    for m in (1, 2, 3):
        f.set_profiling(1)
        got = f.apply(q[:, :m].contiguous(), "fp64")
        passes = 1 if m < 3 else 2
        assert f.last_timings()["main_launches"] >= 2 * passes     # several batches
        assert float((got - ref[:, :m]).abs().max()) <= 1e-13 * scale, m
        assert torch.equal(f.apply(q[:, :m].contiguous(), "fp64"), got)


def test_slots_take_bounded_memory():
    """One more column costs a plan its charges, potentials and partial sums
    (FP64 and FP32) and at most one batch's column of slots."""
    x = W.points_uniform(262144, 3, 97)
    one, two = (SkelFMM(x, "laplace3d", 1e-6, 128, nrhs_max=m, device_build=True).info() for m in (1, 2))
    grown = two["device_bytes"] - one["device_bytes"]
    assert grown <= 2 * 12 * one["n_index"] + 32 * 12 * one["n_work_items"] + BATCH * 32 * 8, grown


@pytest.mark.parametrize("kind,n", [("laplace3d", 40000), ("laplace2d", 30000)])
def test_host_threads_change_no_bit(kind, n):
    """The items, batches and slots are listed by many host threads or one."""
    x = clustered(n, 3 if kind.endswith("3d") else 2, 98)
    q = torch.from_numpy(W.charges_normal(x.shape[0], 2, 99)).cuda()
    one, many = (SkelFMM(x, kind, 1e-6, 64, nrhs_max=2, num_threads=t).apply(q, "fp64") for t in (1, 0))
    assert torch.equal(one, many)
