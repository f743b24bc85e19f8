"""Gradients of a set that holds one group far closer than the rest: what the group's
members feel is larger by orders than what they do to the others, and must not cost
those their digits.

Bars: the ones of the exhaustive tests, 3e-5 sum|grad phi| for FP32 bulk and 1e-12
sum|grad phi| for FP64, each particle against its own sum."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _set(n, members, size):
    rng = np.random.default_rng(n + members)
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.5, 80 + n)
    group = X.mean(axis=0) + np.array([0.11, 0.23, 0.17]) + rng.normal(size=(members, 3)) * size
    return np.ascontiguousarray(np.concatenate([X, group])[rng.permutation(n + members)])


@pytest.mark.parametrize("n,members,size", [(120, 2, 1e-4), (400, 2, 1e-4), (700, 6, 1e-3),
                                            (400, 40, 1e-2)])
def test_gradients(n, members, size):
    X = _set(n, members, size)
    g = inputs.random_weights(len(X), 3)
    Xd, gd = torch.from_numpy(X).cuda(), torch.from_numpy(g).cuda()
    F, S = oracle.forces(X, with_norm=True)
    G, T = oracle.vjp(X, g, with_norm=True)

    def worst(got, ref, scale):
        return float((np.abs(got.cpu().numpy() - ref).max(axis=1) / scale).max())

    assert worst(api.forces(Xd, mode="fp64"), F, S) <= 1e-12
    assert worst(api.forces(Xd, mode="fp32"), F, S) <= 3e-5
    assert worst(api.potential_vjp(Xd, gd, mode="fp32"), G, T) <= 3e-5
    assert worst(api.potential_vjp(Xd, gd, mode="fp64"), G, T) <= 1e-12
