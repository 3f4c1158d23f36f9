"""The quadrature at samples in rho (csrc/series_kernel.cuh) where it can go
wrong: the numbers of samples at which a lane takes one more (32, 64, 96,
128), supports beyond its tables (taken by the per-tap kernel from the list),
windows and supports other than the default, boxes that wrap, and pairs of
visibilities of unequal support.  Against the oracle at the operator's gates,
and against the per-tap kernel, which a plan with a smaller absolute
tolerance uses throughout."""
import math

import numpy as np
import pytest
import torch

import oracle as O
import paper_1903_06555_gb300 as phi
import workloads as W
from tests.test_gpu_parity import gpu_plan, to_t

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "f64": 1e-10}
DT = {"f32": (torch.float32, torch.complex64), "f64": (torch.float64, torch.complex128)}


def observation(geo, jw, n, seed):
    """n baselines of |dw| up to the one that gives support jw in one stack, a
    quarter of them within a box of the grid's edges."""
    uvw = W.uvw_disk(n, 0.4 * geo.Npad * geo.du, 1.0, seed)
    h = 0.5 * geo.Npad * geo.du
    rng = np.random.default_rng(seed)
    q = n // 4
    uvw[:q, 0] = rng.choice([-1, 1], q) * (h - rng.uniform(0.01, 3, q) * geo.du)
    uvw[q // 2:q, 1] = -h + rng.uniform(0.01, 3, q - q // 2) * geo.du
    wm = max(0.0, 0.5 * (jw - geo.J) - 0.25) / geo.c_support
    uvw[:, 2] = np.linspace(-wm, wm, n)[rng.permutation(n)]
    return uvw


# samples per visibility: J_w / sqrt(2) * 4 R intervals and 10 (FP32) or 20
# (FP64) more; supports either side of 32, 64, 96 and 128 of them, and beyond
@pytest.mark.parametrize("precision,jw", [("f32", j) for j in (4, 14, 16, 38, 40, 60, 62, 82, 84, 100)]
                         + [("f64", j) for j in (4, 8, 10, 30, 32, 52, 54, 74, 76, 90)])
def test_supports_match_oracle(precision, jw):
    geo = O.Geometry(64, 2.0, math.radians(20.0), 4.0, tol_rel=1e-13, tol_abs=1e-13)
    n = 12 if jw > 50 else 60
    uvw = observation(geo, jw, n, jw)
    op = O.make_plan(uvw, geo, 1, False, max_support=128)
    assert op.jw.max() == jw
    plan = gpu_plan(uvw, geo, 1, False, precision, max_support=128)
    x, yr = W.point_sources(64, 10, jw), W.random_vis(n, jw)
    rd, cd = DT[precision]
    assert O.rel_l2(plan.degrid(to_t(x, rd)).cpu().numpy(), O.degrid(op, x)) < TOL[precision]
    assert O.rel_l2(plan.grid(to_t(yr, cd)).cpu().numpy(), O.grid(op, yr)) < TOL[precision]
    bad, taps = plan.stats()
    assert bad == 0 and taps == 2 * int((op.jw.astype(np.int64) ** 2).sum())


@pytest.mark.parametrize("mode", ["quadrature", "radial"])
@pytest.mark.parametrize("precision,kw", [
    ("f32", dict(alpha=1.0, support=4, rule="vis", fold=1, det=0)),
    ("f32", dict(alpha=1.5, support=8, rule="stack", fold=0, det=0)),
    ("f32", dict(alpha=1.0, support=6, rule="vis", fold=0, det=1)),
    ("f64", dict(alpha=1.5, support=4, rule="vis", fold=1, det=0)),
    ("f64", dict(alpha=1.0, support=8, rule="stack", fold=1, det=1))])
def test_matches_per_tap_kernels(mode, precision, kw):
    """The same plan with an absolute tolerance below what the samples can
    certify integrates every tap by itself: both within the tolerance of the
    integral, so they agree to it (FP32 rounding 1e-6, or 16-point series in
    radial mode; FP64 1e-12 relative to the largest value)."""
    geo = O.Geometry(128, 2.0, math.radians(15.0), float(kw["support"]), alpha=kw["alpha"])
    uvw = W.uvw_disk(3001, 0.45 * geo.Npad * geo.du, 120.0, 7)
    wts = np.linspace(0.5, 2.0, len(uvw))
    tol = {"f32": (1e-6, 2e-7), "f64": (1e-12, 9e-15)}[precision]
    x, yr = W.random_image(128, 8), W.random_vis(len(uvw), 9)
    rd, cd = DT[precision]
    got = []
    for t in tol:
        p = gpu_plan(uvw, geo, 3, kw["fold"], precision, weights=wts, support_rule=kw["rule"],
                     max_support=128, kernel_mode=mode, grid_deterministic=kw["det"],
                     quad_abs_tol=t, quad_rel_tol=tol[0])
        got.append((p.degrid(to_t(x, rd)).cpu().numpy(), p.grid(to_t(yr, cd)).cpu().numpy()))
    for a, b in zip(*got):
        assert O.rel_l2(a, b) < (5e-6 if precision == "f32" else 1e-11)


def test_results_do_not_depend_on_what_is_sampled_together():
    """Degridding is bitwise the same whether a visibility is sampled with
    its neighbour or alone (a part of the observation, another queue batch)."""
    geo = O.Geometry(128, 2.0, math.radians(20.0), 4.0)
    uvw = W.uvw_disk(60000, 60.0, 40.0, 5)
    x = to_t(W.point_sources(128, 20, 5), torch.float32)
    kw = dict(centres=[0.0], stack_jw=[26])
    whole = gpu_plan(uvw, geo, 1, False, "f32", **kw).degrid(x)
    part = gpu_plan(uvw[7:1200], geo, 1, False, "f32", **kw).degrid(x)
    assert torch.equal(whole[7:1200], part)
