"""Requests that arrive together run together: in a process whose kernels are
loaded and plans warm, with every arrival at once, so that the overlap comes
from the server's slots and not from slow first calls."""
import numpy as np
import pytest

from paper_1903_06555_gb300 import serve as S
from test_gpu_serve import make_requests, run_alone

pytestmark = pytest.mark.gpu


def most_at_once(results):
    edges = sorted([(r.started, 1) for r in results] + [(r.done, -1) for r in results])
    return max(np.cumsum([step for _, step in edges]))


@pytest.mark.parametrize("slots", [1, 4])
def test_warm_requests_overlap_up_to_the_slots(slots):
    reqs = make_requests(seed=3, n=12)
    for r in reqs:
        r.arrival = 0.0
        r.desc = dict(r.desc, grid_deterministic=1)
    alone = [run_alone(r) for r in reqs]           # also loads every kernel they take
    with S.Server(hbm_budget_bytes=1 << 36, slots=slots) as srv:
        got = srv.run_stream(reqs)
    assert all(r.status == "ok" for r in got)
    assert most_at_once(got) == 1 if slots == 1 else 2 <= most_at_once(got) <= slots
    for a, b in zip(alone, got):
        assert np.array_equal(a.y, b.y)
        assert a.dirty is None or np.array_equal(a.dirty, b.dirty)
