"""What a user of this framework has it do, as cases that can be timed and compared.

Every case is the apply phase (u = A q, its transpose, its gradient) on a plan
that the program keeps: the geometry is fixed, as in an iterative solve or a
training step, and each pass brings new charges. `prepare` therefore draws the
charges from the seed and keeps the plan of the geometry it was last asked for.

Fields of a case: the kernel, the number of points n and how they lie, the
right-hand sides, the precision, the tree's leaf size and tolerance, whether
the program called the autotuner, and the call it makes:
  into       apply_into on preallocated column-major buffers
  apply      apply on a row-major (n, nrhs) tensor, a new result each time
  transpose  the same with apply_transpose
  grad       the autograd function, forward and backward
  batch      many point sets as one merged plan, forward and adjoint
"""
import math

import numpy as np
import torch

from paper_2310_16668_gb300 import workloads
from paper_2310_16668_gb300.api import SkelBatch, SkelFMM, skel_apply

COMPLEX = ("helmholtz3d", "helmholtz2d")
LEAF = {"laplace3d": 128, "helmholtz3d": 128, "laplace2d": 64, "helmholtz2d": 64}


def _case(kernel, n, nrhs, precision, call, tuned=False, points="uniform", tol=1e-6, kappa=0.0, sets=0):
    return {"kernel": kernel, "n": n, "nrhs": nrhs, "precision": precision, "call": call, "tuned": tuned,
            "points": points, "leaf": LEAF[kernel], "tol": tol, "kappa": kappa, "sets": sets}


def listed():
    def named(name, *a, **k):
        return {"name": name, **_case(*a, **k)}

    return [
        # the benchmark workload: a million points, 32 right-hand sides at once, tuned once and applied many times
        named("laplace3d 1M rhs32 tuned", "laplace3d", 1 << 20, 32, "fp32_tc", "into", tuned=True),
        # the same kernel as a program calls it that does not tune: a plan straight from the points
        named("laplace3d 256k rhs32", "laplace3d", 1 << 18, 32, "fp32_tc", "into"),
        # adaptive geometry: a surface and a dense cluster, deep tree, boxes of very different sizes
        named("sphere+cluster 256k rhs32", "laplace3d", 1 << 18, 32, "fp32_tc", "into", tuned=True,
              points="sphere_cluster"),
        # odd size, a last pass of right-hand sides that is not full, row-major charges
        named("laplace3d 100003 rhs45", "laplace3d", 100003, 45, "fp32_tc", "transpose"),
        # the default precision: one FP64 product, as a Krylov solver asks for it
        named("laplace3d 128k fp64", "laplace3d", 1 << 17, 1, "fp64", "apply"),
        # the same solver in single precision
        named("laplace3d 64k fp32", "laplace3d", 1 << 16, 1, "fp32", "apply"),
        # a layer of a differentiable program: forward and backward, few columns
        named("laplace3d 20011 rhs8 grad", "laplace3d", 20011, 8, "fp32_tc", "grad"),
        # the smallest calls: a thousand points, where launches count
        named("laplace3d 1000 fp64", "laplace3d", 1000, 1, "fp64", "apply"),
        # the 2D parity workload: 128 x 128 points, tight tolerance, FP64
        named("laplace2d 16k fp64", "laplace2d", 16384, 1, "fp64", "apply", tol=1e-8),
        # complex: scattering in 3D, forward and backward of a real loss
        named("helmholtz3d 64k rhs16 grad", "helmholtz3d", 1 << 16, 16, "fp32_tc", "grad", kappa=25.0),
        # complex: 16 wavelengths across a square, complex64
        named("helmholtz2d 128k rhs8", "helmholtz2d", 1 << 17, 8, "fp32", "into", kappa=100.0),
        # many small boundary curves as one plan, forward and adjoint
        named("curves2d 64 sets rhs4", "laplace2d", 0, 4, "fp32_tc", "batch", tuned=True, points="curves", tol=3e-7,
              sets=64),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | rng.randint(0, 1)

    family = rng.choice(["tc", "tc", "tc", "few", "fp64", "laplace2d", "helmholtz3d", "helmholtz2d", "curves2d"])
    if family == "tc":
        points = rng.choice(["uniform", "uniform", "sphere_cluster"])
        return _case("laplace3d", size(2000, 300000), size(4, 64), "fp32_tc", rng.choice(["into", "apply", "grad"]),
                     tuned=rng.random() < 0.5, points=points)
    if family == "few":
        return _case("laplace3d", size(1000, 200000), rng.randint(1, 3), rng.choice(["fp32", "fp32_tc"]), "apply")
    if family == "fp64":
        return _case("laplace3d", size(1000, 130000), rng.choice([1, 1, 2, 8]), "fp64",
                     rng.choice(["apply", "transpose"]))
    if family == "laplace2d":
        return _case("laplace2d", size(1000, 200000), rng.choice([1, 4, 32]), rng.choice(["fp64", "fp32", "fp32_tc"]),
                     "apply", tol=rng.choice([1e-6, 1e-8]))
    if family == "helmholtz3d":
        return _case("helmholtz3d", size(2000, 130000), size(1, 24), "fp32_tc", rng.choice(["into", "grad"]),
                     kappa=rng.choice([5.0, 25.0]))
    if family == "helmholtz2d":
        return _case("helmholtz2d", size(2000, 200000), rng.choice([1, 4, 8]), rng.choice(["fp32", "fp32_tc"]),
                     rng.choice(["into", "transpose"]), kappa=rng.choice([20.0, 100.0]))
    return _case("laplace2d", 0, rng.choice([4, 8]), "fp32_tc", "batch", tuned=rng.random() < 0.5, points="curves",
                 tol=3e-7, sets=rng.randint(8, 64))


# ---- geometry and plan -----------------------------------------------------------------


def _point_sets(case):
    """The point sets of a case (one, or a batch's), fixed by the case."""
    if case["points"] == "curves":
        sizes = workloads.curve_set_sizes(case["sets"], 4, 1024, 16384)
        return [workloads.points_curve(int(n), 400000 + i) for i, n in enumerate(sizes)]
    if case["points"] == "sphere_cluster":
        return [workloads.points_sphere_cluster(case["n"], 2)]
    return [workloads.points_uniform(case["n"], 2 if case["kernel"].endswith("2d") else 3, 1)]


_kept = {}  # the plan of the last geometry: {key: plan}


def _plan(case):
    key = tuple(case[k] for k in ("kernel", "n", "points", "leaf", "tol", "kappa", "sets", "nrhs", "tuned"))
    if key not in _kept:
        for old in _kept.values():
            old.close()
        _kept.clear()
        sets = _point_sets(case)
        if case["call"] == "batch":
            batch = SkelBatch(sets, case["kernel"], case["tol"], case["leaf"], nrhs_max=case["nrhs"])
            fmm = batch.merged()
            batch.close()
        else:
            fmm = SkelFMM(sets[0], case["kernel"], tol=case["tol"], leaf_size=case["leaf"], kappa=case["kappa"],
                          nrhs_max=case["nrhs"], device_build=True)
        if case["tuned"]:
            fmm.autotune(case["nrhs"])
        _kept[key] = fmm
    return _kept[key]


def _n(case):
    return int(sum(workloads.curve_set_sizes(case["sets"], 4, 1024, 16384))) if case["sets"] else case["n"]


def _charges(case, seed):
    """Charges and cotangents, (nrhs, n): normal, as sources and gradients come."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    dtype = {torch.float64: torch.complex128, torch.float32: torch.complex64}[real] if case["kernel"] in COMPLEX else real
    shape = (case["nrhs"], _n(case))
    return [torch.randn(shape, generator=gen, dtype=dtype, device="cuda") for _ in range(2)]


def prepare(case, seed):
    fmm = _plan(case)
    q, g = _charges(case, seed)
    state = {"fmm": fmm, "call": case["call"], "precision": case["precision"], "nrhs": case["nrhs"]}
    if case["call"] in ("into", "batch"):
        state |= {"q": q, "g": g, "u": torch.empty_like(q), "w": torch.empty_like(q)}
    else:
        state |= {"q": q.t().contiguous(), "g": g.t().contiguous()}
    return state


def run(state):
    fmm, precision = state["fmm"], state["precision"]
    if state["call"] == "into":
        fmm.apply_into(state["q"], state["u"], state["nrhs"], precision)
        return state["u"]
    if state["call"] == "batch":
        fmm.apply_into(state["q"], state["u"], state["nrhs"], precision)
        fmm.apply_into(state["g"], state["w"], state["nrhs"], precision, transpose=True)
        return state["u"], state["w"]
    if state["call"] == "apply":
        return fmm.apply(state["q"], precision)
    if state["call"] == "transpose":
        return fmm.apply_transpose(state["q"], precision)
    q = state["q"].detach().requires_grad_()
    u = skel_apply(q, fmm, precision)
    (grad,) = torch.autograd.grad(u, q, state["g"])
    return u, grad


# ---- what a pass cannot do without ------------------------------------------------------


def work(case):
    """Charges in and potentials out once, the interpolation operators once per direction, and per kernel
    evaluation about 8 operations for the distance and the value plus a multiply-add per right-hand side. The
    evaluations and operator entries per point are those of plans of these trees."""
    n, passes = _n(case), 2 if case["call"] in ("grad", "batch") else 1
    wide = 2 if case["kernel"] in COMPLEX else 1
    size = wide * (8 if case["precision"] == "fp64" else 4)
    flat = case["kernel"].endswith("2d")
    on_curves = case["points"] == "curves"
    pairs = n * min(n / max(1, case["sets"]), 250 if on_curves else 800 if flat else 3000 if case["points"] != "uniform" else 14000)
    operators = n * (10 if on_curves else 40 if flat else 100)
    nbytes = passes * (2 * n * case["nrhs"] + 2 * operators) * size
    return {"bytes": nbytes, "flops": passes * pairs * (8 + 2 * case["nrhs"] * wide * wide)}


# ---- the sums themselves, in 64 bits ----------------------------------------------------


def _kernel(case, d2):
    """Kernel values of squared distances, zero on the diagonal."""
    apart = d2 > 0
    r = torch.where(apart, d2, torch.ones_like(d2)).sqrt()
    if case["kernel"] == "laplace3d":
        g = 1 / (4 * math.pi * r)
    elif case["kernel"] == "laplace2d":
        g = torch.log(r) / (-2 * math.pi)
    elif case["kernel"] == "helmholtz3d":
        g = torch.polar(1 / (4 * math.pi * r), case["kappa"] * r)
    else:
        x = case["kappa"] * r
        g = torch.complex(-torch.special.bessel_y0(x), torch.special.bessel_j0(x)) / 4
    return torch.where(apart, g, torch.zeros_like(g))


def _direct(case, points, charges):
    """sum_j G(x_i, x_j) q_j for each row of charges (nrhs, n)."""
    x = torch.from_numpy(np.ascontiguousarray(points)).cuda()
    n = x.shape[0]
    out = torch.empty_like(charges)
    step = max(1, (1 << 26) // n)
    for i in range(0, n, step):
        d2 = sum((x[i:i + step, None, d] - x[None, :, d]) ** 2 for d in range(x.shape[1]))
        out[:, i:i + step] = charges @ _kernel(case, d2).t()
    return out


def exact(case, seed):
    n, wide = _n(case), 4 if case["kernel"] in COMPLEX else 1
    pairs = n * n if not case["sets"] else n * 16384
    if pairs * (60 + 4 * case["nrhs"]) * wide > 6e12:
        return None
    to = torch.complex128 if case["kernel"] in COMPLEX else torch.float64
    charges = [c.to(to) for c in _charges(case, seed)]
    sets, at = _point_sets(case), 0
    outs = [torch.empty_like(c) for c in charges]
    for points in sets:
        end = at + points.shape[0]
        for c, o in zip(charges, outs):
            o[:, at:end] = _direct(case, points, c[:, at:end].contiguous())
        at = end
    if case["call"] == "batch":
        return tuple(outs)
    if case["call"] == "into":
        return outs[0]
    if case["call"] in ("apply", "transpose"):
        return outs[0].t()
    if case["kernel"] in COMPLEX:  # the gradient is conj(A^T conj(g)); A is symmetric
        outs[1] = _direct(case, sets[0], charges[1].conj().resolve_conj()).conj().resolve_conj()
    return outs[0].t(), outs[1].t()
