"""The complex tensor-core kernel (3D Helmholtz, FP32_TC) across the end of a
group of 128 tiles, where its sums are flushed and its accumulators restart:
single leaves with lists of 128, 129, 130 and 257 tiles, against the complex128
apply of the same plan within 5e-6 of max |u| (the phase kappa r < 44 is an FP32
number, so half a unit in its last place alone is 2e-6 of a far value)."""
import pytest
import torch

from paper_2310_16668_gb300 import SkelFMM
from paper_2310_16668_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_16668_gb300 import build
    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n,tiles", [(4096, 128), (4100, 129), (4160, 130), (8200, 257)])
@pytest.mark.parametrize("nrhs", [16, 19])
def test_groups_match_complex128(n, tiles, nrhs):
    f = SkelFMM(W.points_uniform(n, 3, 81), "helmholtz3d", 1e-6, n, kappa=25.0, nrhs_max=nrhs)
    i = f.info()
    assert i["n_tc_tiles"] == tiles * i["n_tc_items"]
    q = torch.from_numpy(W.charges_complex(n, nrhs, 82)).cuda().to(torch.complex64)
    u = f.apply(q, "fp32_tc")
    f.device_status()
    ref = f.apply(q.to(torch.complex128), "fp64")
    err = (u.to(torch.complex128) - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(err.max()) < 5e-6
    assert torch.equal(f.apply(q, "fp32_tc"), u)
