"""Visibilities that the sampled quadrature (csrc/series_kernel.cuh) does not
settle at its first sampling, and what takes them: one panel more, or the list
of the per-tap and series kernels, for some of a launch's visibilities and for
all of them, plain, under deterministic gridding and under the DDE
convolution; and the per-tap kernels on plans whose absolute tolerance is
below what samples can certify, which is all that still reaches the two-pass
DDE path and the radial DDE boxes.  Against the oracle at the operator's
gates.  Which kernel took what shows in the count of integrand evaluations: a
settled visibility takes 31 per panel and sample, the per-tap kernel 31 per
panel and tap."""
import functools
import math

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from test_gpu_parity import TOL32, TOL64, gpu_plan, to_t

pytestmark = pytest.mark.gpu
TOL = {"f32": TOL32, "f64": TOL64}
DT = {"f32": (torch.float32, torch.complex64), "f64": (torch.float64, torch.complex128)}
# below what the estimate can certify: every visibility as the plan's mode takes it
BELOW = {"f32": 2.4e-7, "f64": 9e-15}


def observation(geo, jw, n, seed, spread=True, edge=False):
    """n baselines, of |dw| up to the one of support jw in one stack (or, with
    spread off, all of that |dw|); with edge, two whose combined boxes cross
    the grid's edge."""
    uvw = W.uvw_disk(n, 0.4 * geo.Npad * geo.du, 1.0, seed)
    wm = max(0.0, 0.5 * (jw - geo.J) - 0.25) / geo.c_support
    w = np.linspace(-wm, wm, n) if spread else np.where(np.arange(n) % 2, wm, -wm)
    uvw[:, 2] = w[np.random.default_rng(seed).permutation(n)]
    if edge:
        h = geo.Npad / 2 * geo.du
        uvw[:2, 0] = [h - 0.4 * geo.du, -h + 0.3 * geo.du]
    return uvw


@functools.lru_cache(maxsize=4)
def case(jw, n, support=4, oversample=2.0, stacks=1, vis=False, taps=0, beta=0.0, **kw):
    """An observation with its DDE kernels (taps > 0) and the oracle's results."""
    geo = O.Geometry(64, oversample, math.radians(20.0), float(support), beta=beta,
                     tol_rel=1e-13, tol_abs=1e-13)
    uvw = observation(geo, jw, n, jw + n, **kw)
    centres = [0.0] if vis else None
    op = O.make_plan(uvw, geo, stacks, False, max_support=128, centres=centres,
                     support_rule=O.SUPPORT_VIS if vis else O.SUPPORT_STACK)
    x, yr = W.point_sources(64, 10, jw), W.random_vis(n, jw)
    if taps:
        dde = W.dde_kernels(n, taps, jw)
        return geo, uvw, op, x, yr, dde, O.degrid_dde(op, x, *dde), O.grid_dde(op, yr, *dde)
    return geo, uvw, op, x, yr, None, O.degrid(op, x), O.grid(op, yr)


def make(c, precision, stacks=1, vis=False, **kw):
    return gpu_plan(c[1], c[0], stacks, False, precision, max_support=128,
                    centres=[0.0] if vis else None, support_rule="vis" if vis else "stack", **kw)


def compare(plan, c, precision):
    """Both directions against the oracle; the evaluations of each."""
    _, _, _, x, yr, dde, y_ref, x_ref = c
    rd, cd = DT[precision]
    xt, yt = to_t(x, rd), to_t(yr, cd)
    y = plan.degrid(xt) if dde is None else plan.degrid_dde(xt, *dde)
    nodes = plan.stats_full(reset=True)[2]
    assert O.rel_l2(y.cpu().numpy(), y_ref) < TOL[precision]
    image = [plan.grid(yt) if dde is None else plan.grid_dde(yt, *dde) for _ in range(2)]
    assert O.rel_l2(image[0].cpu().numpy(), x_ref) < TOL[precision]
    assert plan.stats_full(reset=True)[2] == 2 * nodes
    if plan.desc.grid_deterministic:
        assert torch.equal(*image)
    return nodes


def intervals(geo, jw):
    return int(jw * 0.70710678 * 4.0 * 0.5 * geo.alpha + 1e-3) + 1


# ------------------------------------------------------------- one panel more

# every visibility fails on its one a-priori panel: 12 pixels of support with
# J_w 14 (5.4 of 6 cycles; FP32, 1.5 E = 5e-6 to 8e-6 against 1e-6), 6 pixels with
# J_w 8 (3.3 of 3.4 cycles; FP64, 1e-11 to 9e-11 against 1e-12)
@pytest.mark.parametrize("precision,support,jw", [("f32", 12, 14), ("f64", 6, 8)])
@pytest.mark.parametrize("kind", ["plain", "deterministic", "dde"])
@pytest.mark.parametrize("mode", ["quadrature", "radial"])
def test_failed_visibilities_are_sampled_on_one_panel_more(precision, support, jw, mode, kind):
    c = case(jw, 301, support, taps=5 * (kind == "dde"), spread=False)
    geo, op = c[0], c[2]
    assert np.all(op.jw == jw)
    plan = make(c, precision, kernel_mode=mode, grid_deterministic=int(kind == "deterministic"))
    assert compare(plan, c, precision) == 301 * (intervals(geo, jw) + 1) * 31 * (1 + 2)


def test_a_settled_neighbour_keeps_its_samples():
    """Supports per visibility of 12 (settled on one panel), 14 (not) and 16
    (two panels): those of 12 and 14 are sampled four at a time together, and
    give the same bits as the same baselines alone."""
    c = case(16, 1500, 12, vis=True)
    geo, uvw, op, x = c[:4]
    uvw = uvw.copy()
    uvw[np.random.default_rng(9).random(len(uvw)) < 0.4, 2] = 0.0
    op = O.make_plan(uvw, geo, 1, False, centres=[0.0], support_rule=O.SUPPORT_VIS)
    assert set(op.jw.tolist()) == {12, 14, 16}
    c = (geo, uvw, op, x, c[4], None, O.degrid(op, x), O.grid(op, c[4]))
    plan = make(c, "f32", vis=True)
    panels = {12: 1, 14: 1 + 2, 16: 2}
    assert compare(plan, c, "f32") == sum((intervals(geo, j) + 1) * 31 * panels[j]
                                          for j in op.jw.tolist())
    part = np.nonzero(op.jw == 12)[0][::3]
    alone = make((geo, uvw[part]), "f32", vis=True)
    xt = to_t(x, torch.float32)
    assert np.array_equal(plan.degrid(xt).cpu().numpy()[part], alone.degrid(xt).cpu().numpy())


# ------------------------------------------------------------------ the list

# supports past the tables (FP32 82, FP64 76 pixels at this window) go to the
# list, the others of the same launch are settled
@pytest.mark.parametrize("kind", ["plain", "deterministic", "dde"])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("mode", ["quadrature", "radial"])
def test_some_settled_and_some_left(precision, mode, kind):
    n = 23
    c = case(100 if kind != "dde" else 90, n, vis=True, taps=5 * (kind == "dde"))
    geo, op = c[0], c[2]
    last = {"f32": 118, "f64": 108}[precision]            # intervals the tables hold
    left = np.array([intervals(geo, j) > last for j in op.jw])
    assert 1 < left.sum() < n - 5
    plan = make(c, precision, vis=True, kernel_mode=mode,
                grid_deterministic=int(kind == "deterministic"))
    nodes = compare(plan, c, precision)
    taps = int((op.jw[left].astype(np.int64) ** 2).sum())
    if mode == "quadrature":        # at least one panel's nodes for each tap of the list
        assert nodes > 31 * taps
    # far fewer than by the per-tap kernel throughout (14 panels and more at the
    # largest settled supports)
    assert nodes < 31 * (40 * taps + 14 * sum(intervals(geo, j) + 1 for j in op.jw[~left]))


@pytest.mark.parametrize("precision,tol", [("f32", 2.6e-7), ("f64", 1e-12)])
def test_an_estimate_that_fails_on_another_panel_too_goes_to_the_list(precision, tol):
    """64 pixels of support at oversampling 4 with a taper parameter of 37.3
    (a fifth of the default): 1.5 E is 110 times the tolerance on the four
    a-priori panels and 2.7 times on five (FP64: 80 and 3.5).  This taper falls
    by ten orders over the image; the middle of it is compared."""
    c = case(64, 10, 64, oversample=4.0, beta=37.3)
    _, _, op, _, yr, _, _, x_ref = c
    assert np.all(op.jw == 64)
    x = np.zeros((64, 64))
    x[28:36, 28:36] = W.random_image(8, 30)
    plan = make(c, precision, kb_beta=37.3, quad_abs_tol=tol)
    rd, cd = DT[precision]
    y = plan.degrid(to_t(x, rd)).cpu().numpy()
    assert plan.stats_full()[2] >= 31 * 10 * 64 ** 2
    assert O.rel_l2(y, O.degrid(op, x)) < TOL[precision]
    image = plan.grid(to_t(yr, cd)).cpu().numpy()
    assert O.rel_l2(image[28:36, 28:36], x_ref[28:36, 28:36]) < TOL[precision]


# --------------------------------------------------- below the samples' limit

@pytest.mark.parametrize("jw", [4, 10, 26, 64])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_radial_series_below_the_limit(jw, precision):
    c = case(jw, 12)
    assert c[2].jw.max() == jw
    compare(make(c, precision, kernel_mode="radial", quad_abs_tol=BELOW[precision]), c, precision)


# J_w 38 takes the two-pass path in either mode, 8 the single-pass kernel
@pytest.mark.parametrize("taps", [1, 3, 5, 9])
@pytest.mark.parametrize("jw", [8, 38])
@pytest.mark.parametrize("mode", ["quadrature", "radial"])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_dde_below_the_limit(taps, jw, mode, precision):
    c = case(jw, 40, taps=taps, edge=True)
    assert c[2].jw.max() == jw
    nodes = compare(make(c, precision, kernel_mode=mode, quad_abs_tol=BELOW[precision]), c,
                    precision)
    if mode == "quadrature":
        assert nodes >= 31 * int((c[2].jw.astype(np.int64) ** 2).sum())


@pytest.mark.parametrize("taps", [1, 3, 7, 9, 15])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_dde_of_every_size_from_samples(taps, precision):
    c = case(20, 60, stacks=2, taps=taps, edge=True)
    compare(make(c, precision, stacks=2), c, precision)


# ------------------------------------------------------ per-tap refinement

def test_fp32_refines_like_fp64_where_taps_are_integrated():
    """Supports of 90 pixels, past the tables in both precisions: every tap by
    the per-tap kernel, whose accept and refine decisions from the FP32
    estimate equal those from the FP64 one but for a chunk whose estimate lies
    within the FP32 sums' rounding (1e-7 of 1e-6) of the limit.  One decision
    moves 31 panels' nodes for 64 taps; the bound allows some hundred of the
    12,700 chunks of each direction."""
    geo = O.Geometry(64, 2.0, math.radians(20.0), 4.0)
    n = 100
    uvw = observation(geo, 90, n, 27, spread=False)
    counts = {}
    for precision in ("f32", "f64"):
        plan = gpu_plan(uvw, geo, 1, False, precision, quad_rel_tol=1e-6, quad_abs_tol=1e-6,
                        max_support=128)
        assert plan.info()["max_jw"] == 90
        rd, cd = DT[precision]
        plan.degrid(to_t(W.point_sources(geo.N, 10, 28), rd))
        plan.grid(to_t(W.random_vis(n, 29), cd))
        counts[precision] = plan.stats_full()
    assert counts["f32"][:2] == counts["f64"][:2] == (0, 2 * n * 90 * 90)
    assert abs(counts["f32"][2] - counts["f64"][2]) <= 1e-2 * counts["f64"][2]
