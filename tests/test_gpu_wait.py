"""The bounded waits of the two-pass transforms' column passes
(csrc/fft_kernel.cuh), made to run out by a limit of no polls: the calls come
back, every result computed from the columns left undone is NaN, the plan's
status says so until it is reset, a served request is an error, and the plan
computes as before once it has its limit back."""
import math

import numpy as np
import pytest
import torch

import paper_1903_06555_gb300 as phi
import workloads as W
from paper_1903_06555_gb300 import serve as S

pytestmark = pytest.mark.gpu


def make(n, precision):
    """Three stacks; at 2048 more tiles than blocks."""
    uvw = W.uvw_disk(300, 0.3 * n / math.radians(15.0), 30.0, n)
    tol = 1e-12 if precision == "f64" else 1e-6
    plan = phi.Plan(torch.from_numpy(uvw), image_n=n, fov_rad=math.radians(15.0), n_stacks=3,
                    precision=precision, quad_rel_tol=tol, quad_abs_tol=tol, grid_deterministic=1)
    assert plan.info()["n_dropped"] == 0
    x = torch.from_numpy(W.random_image(n, 1)).to("cuda", plan.real_dtype)
    y = torch.from_numpy(W.random_vis(len(uvw), 2)).to("cuda", plan.complex_dtype)
    return plan, x, y


@pytest.mark.parametrize("polls", [0, 1])
@pytest.mark.parametrize("n,precision", [(64, "f32"), (256, "f32"), (512, "f64"), (2048, "f32")])
def test_a_wait_that_runs_out_shows_in_results_and_status(n, precision, polls):
    plan, x, y = make(n, precision)
    vis, image = plan.degrid(x), plan.grid(y)
    for call, arg, want in ((plan.degrid, x, vis), (plan.grid, y, image)):
        plan.set_wait_limit(polls)
        got = call(arg)
        torch.cuda.synchronize()
        lost = torch.isnan(torch.view_as_real(got).sum(-1) if got.is_complex() else got)
        assert torch.equal(got[~lost], want[~lost])
        if polls == 0:
            assert bool(lost.all())
        if bool(lost.any()):
            with pytest.raises(phi.PhiError) as e:
                plan.stats()
            assert e.value.status == phi.PHI_ERR_TIMEOUT
        plan.set_wait_limit()
        try:
            plan.stats(reset=True)
        except phi.PhiError:
            pass
        assert torch.equal(call(arg), want)
        plan.stats()
    plan.close()


def test_a_served_request_whose_transform_gave_up_is_an_error(monkeypatch):
    class Impatient(phi.Plan):
        def __init__(self, *a, **kw):
            super().__init__(*a, **kw)
            self.set_wait_limit(0)

    uvw = W.uvw_disk(500, 20.0, 10.0, 3)
    desc = dict(image_n=64, fov_rad=math.radians(20.0), n_stacks=2)
    req = S.Request(0, uvw, desc, image=np.ones((64, 64)), ops=("degrid", "grid"))
    for cls, status in ((Impatient, "error"), (phi.Plan, "ok")):
        monkeypatch.setattr(S, "Plan", cls)
        with S.Server(hbm_budget_bytes=1 << 34, slots=1) as srv:
            res = srv.run_stream([req], realtime=False)[0]
        assert res.status == status
        if status == "error":
            assert "wait" in res.error and res.y is None and res.dirty is None
        else:
            assert np.isfinite(res.y).all() and np.isfinite(res.dirty).all()
