"""The chirp transforms (csrc/czt_kernel.cuh) at sizes with large prime factors,
either side of each length of their convolution and beside the sizes they take
(378, 524, 614: the library's), several stacks and more than one group of them,
against the oracle at the operator's gates."""
import math

import pytest
import torch

import oracle as O
import workloads as W
from tests.test_gpu_parity import gpu_plan, to_t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [378, 382, 508, 524, 548, 582, 614, 842, 1018, 1090, 1986, 2042])
def test_sizes_match_oracle(n):
    geo = O.Geometry(n, 2.0, math.radians(15.0), 4.0, tol_rel=1e-13, tol_abs=1e-13)
    k = 3 if n <= 582 else 1
    uvw = W.uvw_disk(40, 0.45 * geo.Npad * geo.du, 20.0, n)
    op = O.make_plan(uvw, geo, k, True)
    # three stacks in groups of one or two grids
    plan = gpu_plan(uvw, geo, k, True, "f32", max_grid_mib=max(1, 20 * geo.Npad ** 2 >> 20))
    x, yr = W.random_image(n, 1), W.random_vis(len(uvw), 2)
    assert O.rel_l2(plan.degrid(to_t(x, torch.float32)).cpu().numpy(), O.degrid(op, x)) < 1e-5
    assert O.rel_l2(plan.grid(to_t(yr, torch.complex64)).cpu().numpy(), O.grid(op, yr)) < 1e-5
