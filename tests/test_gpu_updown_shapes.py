"""Launch shapes of the FP32 upward / downward passes: all give the same bits,
and what tuning changes."""
import pytest
import torch

from paper_2310_16668_gb300 import SkelFMM, _lib
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


@pytest.mark.parametrize("nrhs", [1, 4, 8])
def test_tuning_for_few_columns(nrhs):
    """Up to 8 columns the tuner has shapes to choose from (a row or a column
    per lane), no choice is slower than the default, and neither their bits nor
    those of wider applies change."""
    f = SkelFMM(clustered(12000, 3, 41), "laplace3d", 1e-6, 16, nrhs_max=40)
    q = torch.from_numpy(W.charges_normal(15000, 40, 42)).cuda().float()
    few = q[:, :nrhs].contiguous()
    ref, ref_few = f.apply(q, "fp32"), f.apply(few, "fp32")
    rep = f.autotune(nrhs, allow_store=False)
    assert rep["n_updown"] > 0 and 0 < rep["ms_updown_tuned"] <= rep["ms_updown_default"] + 1e-9
    assert torch.equal(f.apply(q, "fp32"), ref) and torch.equal(f.apply(few, "fp32"), ref_few)


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("kind", ["laplace3d", "laplace2d"])
def test_launch_shapes_same_bits_for_few_columns(nrhs, kind):
    """The kernels with a row per lane (33, 40) and with a column per lane add
    the same partial sums in the same order."""
    lib = _lib.load()
    x = clustered(9000, int(kind[-2]), 43)
    f = SkelFMM(x, kind, 1e-8, 50, nrhs_max=8)
    q = torch.from_numpy(W.charges_normal(x.shape[0], nrhs, 44)).cuda().float()
    ref = [fn(q, "fp32") for fn in (f.apply, f.apply_transpose)]
    for code in (1, 2, 4, 8, 17, 18, 20, 24, 33, 40):
        _lib.check(lib.skel_test_set_updown(f._h, code))
        for fn, r in zip((f.apply, f.apply_transpose), ref):
            assert torch.equal(fn(q, "fp32"), r), code


@pytest.mark.parametrize("nrhs", [9, 11, 37])
@pytest.mark.parametrize("precision", ["fp32", "fp32_tc"])
def test_launch_shapes_same_bits_at_odd_widths(nrhs, precision):
    """Every launch shape at widths above 8 that are no multiple of 4 (the
    4-byte copies of the asynchronous-copy kernel) against the default rule's
    bits, plain and transposed."""
    lib = _lib.load()
    x = clustered(12000, 3, 41)
    f = SkelFMM(x, "laplace3d", 1e-6, 16, nrhs_max=40)
    q = torch.from_numpy(W.charges_normal(x.shape[0], nrhs, 42)).cuda().float()
    ref = [fn(q, precision) for fn in (f.apply, f.apply_transpose)]
    for code in (1, 2, 4, 8, 17, 18, 20, 24):
        _lib.check(lib.skel_test_set_updown(f._h, code))
        for fn, r in zip((f.apply, f.apply_transpose), ref):
            assert torch.equal(fn(q, precision), r), code
        f.device_status()
