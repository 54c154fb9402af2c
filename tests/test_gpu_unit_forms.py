"""The forms into which the on-the-fly tensor-core translations are divided,
each reached by construction (the division is asked for, so that a changed rule
cannot silently take the coverage away), every column against the FP64 apply of
the same plan within 2e-6 of max |u|, the bound the tensor-core path is held to
elsewhere."""
import ctypes

import pytest
import torch

from paper_2310_16668_gb300 import SkelBatch, SkelFMM, _lib
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


def _units(f):
    """CTAs with one item, sharing two, with two unrelated ones; cut items; longest piece."""
    out = (ctypes.c_int64 * 5)()
    _lib.check(_lib.load().skel_test_units(f._h, ctypes.cast(out, ctypes.c_void_p)))
    return dict(zip(("single", "shared", "unrelated", "cut", "longest"), out))


def _check(f, n, nrhs, seed):
    q = torch.from_numpy(W.charges_normal(n, nrhs, seed)).cuda().float()
    u = f.apply(q, "fp32_tc")
    f.device_status()
    ref = f.apply(q.double(), "fp64")
    err = (u.double() - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(err.max()) < 2e-6
    assert torch.equal(f.apply(q, "fp32_tc"), u)
    return q, u


@pytest.mark.parametrize("n,leaf,dist", [(500, 500, "uniform"), (513, 513, "uniform"), (3000, 128, "uniform"),
                                         (7000, 128, "uniform"), (3500, 40, "clustered")])
@pytest.mark.parametrize("nrhs", [4, 33])
def test_small_plans_are_cut_into_short_pieces(n, leaf, dist, nrhs):
    """3D plans with few tiles: no piece is longer than 16 tiles (lists of 16
    and 17 tiles, ragged last pieces), and the stored kernels, which do not cut,
    give the same bits."""
    x = W.points_uniform(n, 3, 71) if dist == "uniform" else clustered(n, 3, 71)
    n = x.shape[0]
    f = SkelFMM(x, "laplace3d", 1e-6, leaf, nrhs_max=nrhs)
    un = _units(f)
    assert un["longest"] == 16 and un["shared"] == un["unrelated"] == 0
    assert (un["cut"] > 0) == (n != 500)
    q, u = _check(f, n, nrhs, 72)
    for stages in (4, 5, 8):
        g = SkelFMM(x, "laplace3d", 1e-6, leaf, nrhs_max=nrhs, store_tiles=1, store_stages=stages)
        assert torch.equal(g.apply(q, "fp32_tc"), u), stages


def test_merged_plans_keep_their_sets_segments():
    """A small and a larger set in one plan: each gets its own plan's bits."""
    sets = [W.points_uniform(n, 3, 73 + n) for n in (1500, 30000, 3000)]
    nrhs = 5
    b = SkelBatch(sets, "laplace3d", 1e-6, 128, nrhs_max=nrhs)
    m = b.merged()
    q = torch.randn((nrhs, m.n), generator=torch.Generator("cuda").manual_seed(74), device="cuda")
    u = torch.empty_like(q)
    m.apply_into(q, u, nrhs, "fp32_tc")
    m.device_status()
    for i, f in enumerate(b.plans):
        at = slice(b.offsets[i], b.offsets[i] + len(sets[i]))
        one = torch.empty((nrhs, len(sets[i])), device="cuda")
        f.apply_into(q[:, at].contiguous(), one, nrhs, "fp32_tc")
        assert torch.equal(one, u[:, at]), i


@pytest.mark.parametrize("kind,n,leaf,form", [
    ("laplace3d", 30000, 128, "pairs, cut"),
    ("laplace3d", 20000, 20000, "pairs, cut"),           # one leaf: 157 items, the last one of 32 rows
    ("laplace3d", 20011, 128, "pairs, pieces of 32"),
    ("laplace3d", 12000, 128, "single, pieces of 32"),
    ("laplace3d", 120000, 128, "pieces of two segments"),
    ("laplace3d", 150000, 128, "pairs, whole lists"),    # the form of every larger 3D plan
    ("laplace2d", 4300, 4300, "single, cut"),
])
@pytest.mark.parametrize("nrhs", [4, 33])
def test_forms_match_fp64(kind, n, leaf, form, nrhs):
    x = W.points_uniform(n, int(kind[-2]), 75)
    f = SkelFMM(x, kind, 1e-6, leaf, nrhs_max=nrhs, device_build=n > 60000)
    un = _units(f)
    if form.startswith("single"):
        assert un["single"] > 0 and un["cut"] > 0 and un["shared"] == un["unrelated"] == 0
        assert un["longest"] == (32 if "32" in form else 128)
    else:
        assert un["shared"] > 0 and un["unrelated"] > 0
        if form == "pairs, cut":
            assert un["cut"] > 0 and un["longest"] == 128
        elif form == "pairs, pieces of 32":
            assert un["cut"] > 0 and un["longest"] == 32
        elif form == "pieces of two segments":
            assert un["cut"] > 0 and un["longest"] == 256
        else:
            assert un["cut"] == 0 and un["longest"] > 256
    _check(f, n, nrhs, 76)
