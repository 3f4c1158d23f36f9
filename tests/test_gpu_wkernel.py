"""Kernel values either side of the point count where a point goes from 16
lanes to 4: the same nodes summed in another order."""
import math

import pytest
import torch

import paper_1903_06555_gb300 as phi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [-1, 0, 17])
def test_values_do_not_depend_on_the_point_count(extra):
    uvw = torch.zeros(1, 3, dtype=torch.float64)
    with phi.Plan(uvw, image_n=256, fov_rad=math.radians(20.0), n_stacks=1) as plan:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        n = 640 * sms + extra
        g = torch.Generator().manual_seed(11)
        rho = 24.0 * torch.rand(n, generator=g, dtype=torch.float64)
        dw = 60.0 * (2.0 * torch.rand(n, generator=g, dtype=torch.float64) - 1.0)
        rho[:8] = torch.tensor([0.0, 1e-9, 0.5, 0.95, 1.0, 1.5, 2.0, 24.0], dtype=torch.float64)
        k, bad = plan.wkernel(rho, dw)
        parts = [plan.wkernel(rho[i:i + 40009], dw[i:i + 40009]) for i in range(0, n, 40009)]
        # g is positive, so K(0, 0) is the sum of the terms' magnitudes.  Four
        # lanes add 4 terms a panel one after another, at most 12 panels at
        # these radii and offsets, and 4 partial sums: 52 roundings of at most
        # 2^-24 of that sum, and fewer for 16 lanes.
        scale = float(plan.wkernel([0.0], [0.0])[0].abs())
    whole = torch.cat([p[0] for p in parts])
    assert bad == sum(p[1] for p in parts) == 0
    assert float((k - whole).abs().max()) <= 2 * 52 * 2.0 ** -24 * math.sqrt(2.0) * scale
