"""The server's HBM budget against what its slots really hold on the device: exhaustive
forces and FP64 requests, whose fast paths take gigabytes, shrink to it or take the triple
sweep, and idle slots give their buffers back when others need the room."""
import numpy as np
import pytest
import torch

from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu

SLACK = 8 << 20  # allocation granularity of the buffers a request takes


def _held(free0):
    torch.cuda.synchronize()
    return free0 - torch.cuda.mem_get_info()[0]


def _run(srv, reqs):
    """Every request's result; a minute is far more than any takes."""
    tickets = [srv.submit(**r) for r in reqs]
    out = []
    for t in tickets:
        st, res, o = srv.poll(t, timeout_us=60_000_000)
        assert st == 0, res
        out.append(o)
    return out


def _alone(r):
    X = torch.from_numpy(r["X"]).cuda()
    f = api.forces if r["kind"] == "forces" else api.potential
    return f(X, mode=r["mode"]).cpu().numpy()


@pytest.mark.parametrize("budget_mb", [2, 64])
def test_small_budget(budget_mb):
    reqs = [dict(X=inputs.uniform_cube(n, n ** (1 / 3), 0.4, n), kind=kind, mode=mode)
            for n, kind, mode in ((4096, "forces", "fp32"), (2000, "potential", "fp64"),
                                  (1500, "forces", "fp64"), (700, "forces", "fp32"))]
    want = [_alone(r) for r in reqs]
    torch.cuda.empty_cache()
    srv = api.Server(0, hbm_budget_bytes=budget_mb << 20, slots=2)
    _run(srv, [dict(X=reqs[0]["X"][:10], kind="potential", mode="fp64")] * 4)
    free0 = torch.cuda.mem_get_info()[0]
    got = _run(srv, reqs)
    assert _held(free0) <= (budget_mb << 20) + SLACK
    assert srv.stats()["reserved_bytes"] <= budget_mb << 20
    for r, a, b in zip(reqs, got, want):
        tol = 1e-12 if r["mode"] == "fp64" else 3e-6
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
    srv.close()


def test_idle_slots_make_room():
    """Each of these takes most of the budget, whichever slot runs it."""
    X = inputs.uniform_cube(6000, 18.2, 0.4, 5)
    big = dict(X=X, kind="forces", mode="fp32")
    wide = dict(X=X[:3500], kind="potential", mode="fp64")
    want = [_alone(big), _alone(wide)]
    torch.cuda.empty_cache()
    budget = 3 << 30
    srv = api.Server(0, hbm_budget_bytes=budget, slots=3)
    _run(srv, [dict(X=X[:10], kind="potential", mode="fp64")] * 6)
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        got = _run(srv, [big, wide, big, big, wide])
        assert _held(free0) <= budget + SLACK
        assert srv.stats()["reserved_bytes"] <= budget
    for a, b in zip(got, (want[0], want[1], want[0], want[0], want[1])):
        assert np.linalg.norm(a - b) <= 1e-9 * np.linalg.norm(b)
    srv.close()
