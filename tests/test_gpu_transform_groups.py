"""Several stacks and several groups of them through every transform, in both
precisions: the two-pass transforms at each of their sizes (the tiles' grid
coordinate, tiles of one grid followed by tiles of the next, the sum over the
stacks and over the groups), the chirp transforms at each of their lengths,
small images with many stacks (whose adjoint rows split the stacks over sets
of threads), and the library's transforms beside them in batches with a grid
left over.  Against the oracle at the operator's gates."""
import functools
import math

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from test_gpu_parity import gpu_plan, to_t

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "f64": 1e-10}
DT = {"f32": (torch.float32, torch.complex64), "f64": (torch.float64, torch.complex128)}


@functools.lru_cache(maxsize=2)
def case(n, k):
    geo = O.Geometry(n, 2.0, math.radians(15.0), 4.0, tol_rel=1e-13, tol_abs=1e-13)
    uvw = W.uvw_disk(max(40, 8 * k), 0.45 * geo.Npad * geo.du, 5.0 * k, n)
    op = O.make_plan(uvw, geo, k, True)
    x, yr = W.random_image(n, 1), W.random_vis(len(uvw), 2)
    return geo, uvw, x, yr, O.degrid(op, x), O.grid(op, yr)


def transform(n, precision):
    """What takes grids of 2 n, at the sizes used here."""
    if n in (512, 1024, 2048) or (precision == "f32" and n in (64, 128, 256)):
        return "two-pass"
    return "chirp" if precision == "f32" and n in (498, 842, 1018, 1090, 1986) else "library"


def check(n, k, precision, group, mib):
    geo, uvw, x, yr, y_ref, x_ref = case(n, k)
    plan = gpu_plan(uvw, geo, k, True, precision, max_grid_mib=mib, max_support=128)
    info = plan.info()
    assert plan.transform() == transform(n, precision)
    assert info["group"] == group and sum(c > 0 for c in info["counts"]) == k
    rd, cd = DT[precision]
    assert O.rel_l2(plan.degrid(to_t(x, rd)).cpu().numpy(), y_ref) < TOL[precision]
    assert O.rel_l2(plan.grid(to_t(yr, cd)).cpu().numpy(), x_ref) < TOL[precision]
    plan.close()


def grid_mib(n, precision):
    return 4 * n * n * (16 if precision == "f64" else 8) / 2 ** 20


# two-pass transforms, 128 to 2048; chirp transforms of length 1024 (498),
# 2048 (842, 1018) and 4096 (1090, 1986); the library's (500, 1000)
@pytest.mark.parametrize("n", [128, 256, 500, 498, 512, 842, 1000, 1018, 1024, 1090, 1986, 2048])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_groups_of_two_and_one(n, precision):
    check(n, 3, precision, 2, max(1, math.ceil(2 * grid_mib(n, precision))))


# 64^2: eight grids of FP32 to a MiB
@pytest.mark.parametrize("n,k,group,mib", [
    (64, 9, 5, 1), (64, 20, 7, 1),           # groups of 5 + 4, and of 7 + 7 + 6
    (64, 2, 2, 0), (64, 3, 3, 0), (64, 8, 8, 0), (64, 13, 13, 0), (64, 40, 40, 0),
    (128, 2, 2, 0), (128, 24, 24, 0), (256, 5, 5, 0), (256, 20, 10, 20)])
def test_small_images_with_many_stacks(n, k, group, mib):
    check(n, k, "f32", group, mib)


@pytest.mark.parametrize("n,k", [(70, 24), (640, 3), (644, 3)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_blocks_of_the_image_step(n, k, precision):
    """Grids narrower and wider than the image step's change of block (FP32,
    Npad 1280), and fewer rows than it launches blocks for large ones."""
    check(n, k, precision, k, 0)


def test_library_batches_with_a_grid_left_over():
    """35 grids of 2000^2 exceed one batch of at most 1 GiB: two batches of 17
    and one grid by itself, against the same stacks one grid at a time."""
    geo = O.Geometry(1000, 2.0, math.radians(15.0), 4.0)
    k = 35
    uvw = W.uvw_disk(8 * k, 0.45 * geo.Npad * geo.du, 5.0 * k, 7)
    x, yr = W.random_image(1000, 1), W.random_vis(len(uvw), 2)
    got = []
    for mib, group in ((0, k), (1, 1)):
        plan = gpu_plan(uvw, geo, k, True, "f32", max_grid_mib=mib, max_support=128)
        assert plan.info()["group"] == group
        got.append((plan.degrid(to_t(x, torch.float32)).cpu().numpy(),
                    plan.grid(to_t(yr, torch.complex64)).cpu().numpy()))
        plan.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and O.rel_l2(a, b) < 2e-6
