"""The two-pass image-domain transforms (csrc/fft_kernel.cuh) at every size they
take and beside it (cuFFT takes the neighbours), several stacks and more than
one group of them, against the oracle at the operator's gates."""
import math

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from tests.test_gpu_parity import gpu_plan, to_t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n", [62, 64, 66, 128, 256, 512, 1024, 2048])
def test_sizes_match_oracle(n, precision):
    geo = O.Geometry(n, 2.0, math.radians(15.0), 4.0, tol_rel=1e-13, tol_abs=1e-13)
    k = 3 if n <= 256 else 1
    uvw = W.uvw_disk(40, 0.45 * geo.Npad * geo.du, 20.0, n)
    op = O.make_plan(uvw, geo, k, True)
    # three stacks in groups of one or two grids
    grid = geo.Npad ** 2 * (16 if precision == "f64" else 8)
    plan = gpu_plan(uvw, geo, k, True, precision, max_grid_mib=max(1, int(2.5 * grid) >> 20))
    x, yr = W.random_image(n, 1), W.random_vis(len(uvw), 2)
    rd, cd, tol = (torch.float64, torch.complex128, 1e-10) if precision == "f64" else \
        (torch.float32, torch.complex64, 1e-5)
    assert O.rel_l2(plan.degrid(to_t(x, rd)).cpu().numpy(), O.degrid(op, x)) < tol
    assert O.rel_l2(plan.grid(to_t(yr, cd)).cpu().numpy(), O.grid(op, yr)) < tol


def test_other_oversampling_takes_the_library_transform():
    geo = O.Geometry(128, 1.5, math.radians(15.0), 6.0, tol_rel=1e-13, tol_abs=1e-13)
    uvw = W.uvw_disk(40, 0.45 * geo.Npad * geo.du, 20.0, 3)
    op = O.make_plan(uvw, geo, 1, False)
    x = W.random_image(128, 1)
    plan = gpu_plan(uvw, geo, 1, False, "f32")
    assert O.rel_l2(plan.degrid(to_t(x, torch.float32)).cpu().numpy(), O.degrid(op, x)) < 1e-5
