"""Sets that the contractions give back to the triple sweeps on the device: too many
near pairs, or a pair that the packed points do not resolve. They are solved as the sweep
solves them: gradients equal to those of a context without room for a contraction,
potentials from a pair table, with the FP64 coordinates' accuracy."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


def test_too_many_near_pairs():
    """400 points on two sites: every cross pair is near. (Coincident pairs are left out
    of gradients, which do not report them.)"""
    X = np.zeros((400, 3))
    X[::2, 0] = 1.5
    X[200:] += np.array([0.0, 0.25, 0.5]) * (np.arange(200) % 2)[:, None]
    Xd, g = _dev(X), _dev(inputs.random_weights(400, 9))
    sweep = api.Context(0, 1 << 20)
    for call in (lambda c: api.forces(Xd, mode="fp32", ctx=c),
                 lambda c: api.forces(Xd, mode="fp64", ctx=c),
                 lambda c: api.potential_vjp(Xd, g, mode="fp32", ctx=c)):
        got, want = call(None).cpu().numpy(), call(sweep).cpu().numpy()
        assert np.all(np.isfinite(want)) and np.linalg.norm(want) > 0
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    sweep.close()
    with pytest.raises(Exception) as e:
        api.potential(_dev(np.concatenate([X] * 4)), mode="fp32")
    assert getattr(e.value, "status", None) == -1


@pytest.mark.parametrize("n", [1300, 3001])
def test_unresolved_pair_far_from_the_origin(n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.4, 44) + 1.23456789e9
    X[7] = X[9]
    for _ in range(8):
        X[7, 2] = np.nextafter(X[7, 2], 2e9)  # 2e-6 apart
    idx = np.unique(np.concatenate([inputs.sample_indices(n, 40, 8), [7, 9]]))
    got = api.potential(_dev(X), mode="fp32").cpu().numpy()[idx]
    assert np.all(np.abs(got - oracle.phi(X, idx)) <= 3e-6 * oracle.phi_parts(X, idx))
