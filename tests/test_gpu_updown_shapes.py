"""Launch shapes of the FP32 upward / downward passes: where there is a choice
and where there is none."""
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
def test_autotune_has_no_shape_to_choose_for_few_columns(nrhs):
    """Up to 8 columns run one kernel in one shape: nothing is timed, and
    nothing a wider apply would use is set from noise."""
    f = SkelFMM(clustered(12000, 3, 41), "laplace3d", 1e-6, 16, nrhs_max=40)
    wide = f.autotune(9, allow_store=False)
    assert wide["n_updown"] > 0 and wide["ms_updown_tuned"] > 0
    rep = f.autotune(nrhs, allow_store=False)
    assert (rep["n_updown"], rep["n_changed"], rep["ms_updown_default"], rep["ms_updown_tuned"]) == (0, 0, 0.0, 0.0)


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
