"""The FP32 contraction at any unit of length, offset and weight: its bars are those of
the exhaustive tests at spacing 1 (3e-6 sum|phi|, 3e-5 sum|grad phi|), whatever power of
two the points are scaled by, and one far point does not touch the others."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


def _phi_ok(X, got, idx):
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    return np.all(np.abs(got[idx] - ref) <= 3e-6 * ref_abs)


@pytest.mark.parametrize("k", [-40, -30, -14, -7, 7, 14, 22, 34, 60])
def test_powers_of_two(k):
    X = inputs.uniform_cube(1300, 1300 ** (1 / 3), 0.4, 41)
    idx = inputs.sample_indices(1300, 48, 4)
    got = np.ldexp(api.potential(_dev(np.ldexp(X, k)), mode="fp32").cpu().numpy(), 9 * k)
    assert _phi_ok(X, got, idx)
    X = X[:300]
    g = inputs.random_weights(300, 5)
    F, S = oracle.forces(X, with_norm=True)
    G, T = oracle.vjp(X, g, with_norm=True)
    Xd = _dev(np.ldexp(X, k))
    got = np.ldexp(api.forces(Xd, mode="fp32").cpu().numpy(), 10 * k)
    assert np.all(np.abs(got - F).max(axis=1) <= 3e-5 * S)
    for w in (0, 90, -90):  # weights have a unit of their own
        got = api.potential_vjp(Xd, _dev(np.ldexp(g, w)), mode="fp32").cpu().numpy()
        assert np.all(np.abs(np.ldexp(got, 10 * k - w) - G).max(axis=1) <= 3e-5 * T)


@pytest.mark.parametrize("far", [1e3, 1e5, 1e8, 1e10])
def test_one_far_point(far):
    X = inputs.uniform_cube(1300, 1300 ** (1 / 3), 0.4, 42)
    X[700] = far
    idx = np.setdiff1d(inputs.sample_indices(1300, 48, 6), [700])
    got = api.potential(_dev(X), mode="fp32").cpu().numpy()
    assert np.all(np.isfinite(got)) and _phi_ok(X, got, idx)
    X = X[600:900]
    F, S = oracle.forces(X, with_norm=True)
    got = api.forces(_dev(X), mode="fp32").cpu().numpy()
    others = np.arange(300) != 100
    assert np.all(np.abs(got - F).max(axis=1)[others] <= 3e-5 * S[others])


@pytest.mark.parametrize("off", [1e4, 1e8, 1e9])
def test_offset(off):
    """Coordinates are taken relative to a point of the set before they are rounded."""
    X = inputs.uniform_cube(1300, 1300 ** (1 / 3), 0.4, 43) + off
    assert _phi_ok(X, api.potential(_dev(X), mode="fp32").cpu().numpy(),
                   inputs.sample_indices(1300, 48, 7))
    X = X[:300]
    F, S = oracle.forces(X, with_norm=True)
    got = api.forces(_dev(X), mode="fp32").cpu().numpy()
    assert np.all(np.abs(got - F).max(axis=1) <= 3e-5 * S)
