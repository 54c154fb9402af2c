"""The complex tensor-core kernel (3D Helmholtz, FP32_TC) where its sums and
masks change: lists shorter than a pair of tiles, one tile more than a group,
ragged chunks, touching leaves with masked sources, and right-hand sides that
end inside a pass of 16. Every column against the complex128 apply of the same
plan within 5e-6 of max |u|: the phase kappa r < 44 is an FP32 number, so half
a unit in its last place alone is 2e-6 of a far value."""
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


@pytest.mark.parametrize("n,leaf,dist", [
    (5, 8, "uniform"),
    (97, 100, "uniform"),                      # a pair, a whole and a ragged tile
    (530, 530, "uniform"),                     # 17 tiles: a group of 16 and one more
    (3001, 48, "uniform"),
    (4000, 20, "clustered"),
])
@pytest.mark.parametrize("nrhs", [16, 19])
def test_complex_units_match_complex128(n, leaf, dist, nrhs):
    x = W.points_uniform(n, 3, 81) if dist == "uniform" else clustered(n, 3, 81)
    f = SkelFMM(x, "helmholtz3d", 1e-6, leaf, kappa=25.0, nrhs_max=nrhs)
    q = torch.from_numpy(W.charges_complex(x.shape[0], nrhs, 82)).cuda().to(torch.complex64)
    u = f.apply(q, "fp32_tc")
    f.device_status()
    ref = f.apply(q.to(torch.complex128), "fp64")
    err = (u.to(torch.complex128) - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(err.max()) < 5e-6
    assert torch.equal(f.apply(q, "fp32_tc"), u)
