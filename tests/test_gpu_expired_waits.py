"""Waits of the tensor-core kernels that run out (a context switch makes them): the
kernels end on their own, with nothing in flight, the context stays usable, and the
solve is done again by the triple sweep."""
import numpy as np
import pytest
import torch

from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu

CALLS = {
    "phi32": (1500, lambda X, g, c: api.potential(X, mode="fp32", ctx=c)),
    "phi64": (700, lambda X, g, c: api.potential(X, mode="fp64", ctx=c)),
    "forces32": (700, lambda X, g, c: api.forces(X, mode="fp32", ctx=c)),
    "forces64": (500, lambda X, g, c: api.forces(X, mode="fp64", ctx=c)),
    "vjp32": (700, lambda X, g, c: api.potential_vjp(X, g, mode="fp32", ctx=c)),
}


def _case(name):
    n, call = CALLS[name]
    X = torch.from_numpy(inputs.uniform_cube(n, n ** (1 / 3), 0.4, 70 + n)).cuda()
    g = torch.from_numpy(inputs.random_weights(n, 71 + n)).cuda()
    return X, g, call


@pytest.mark.parametrize("name", sorted(CALLS))
def test_context_stays_usable(name):
    X, g, call = _case(name)
    want = call(X, g, None).cpu().numpy()
    ctx = api.Context(0)
    for _ in range(3):
        ctx.expire_waits(True)
        call(X, g, ctx)
        ctx.expire_waits(False)
        got = call(X, g, ctx).cpu().numpy()
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    ctx.close()


@pytest.mark.parametrize("name", sorted(CALLS))
def test_result_is_right(name):
    """Whatever the contraction left behind: the sweep's own accuracy."""
    X, g, call = _case(name)
    want = call(X, g, None).cpu().numpy()
    ctx = api.Context(0)
    ctx.expire_waits()
    for _ in range(3):
        got = call(X, g, ctx).cpu().numpy()
        tol = 1e-12 if name.endswith("64") else 3e-6
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
    ctx.close()
