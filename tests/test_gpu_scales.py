"""Exhaustive sums do not depend on the unit of length: phi is homogeneous of degree
-9 and its gradient of degree -10, so a set scaled by a power of two has the same
results times an exact power of two, over the FP64 range of spacings. A set that spans
more orders than the packed points resolve is solved by the triple sweep.

Bars: 1e-12 |Phi| and 1e-12 sum|grad phi| in FP64 (the exhaustive tests' bars)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


@pytest.mark.parametrize("n", [200, 400])
@pytest.mark.parametrize("k", [-66, -60, -45, -3, 0, 45, 60, 66])
def test_fp64_powers_of_two(n, k):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.4, 30 + n)
    phi = oracle.phi(X)
    got = np.ldexp(api.potential(_dev(np.ldexp(X, k)), mode="fp64").cpu().numpy(), 9 * k)
    assert np.all(np.abs(got - phi) <= 1e-12 * np.abs(phi))
    F, S = oracle.forces(X, with_norm=True)
    got = np.ldexp(api.forces(_dev(np.ldexp(X, k)), mode="fp64").cpu().numpy(), 10 * k)
    assert np.all(np.abs(got - F).max(axis=1) <= 1e-12 * S)


@pytest.mark.parametrize("scale", [1e-20, 1e-15, 1e-13, 1e13, 1e15, 1e20])
def test_fp64_spacings(scale):
    X = inputs.uniform_cube(300, 300 ** (1 / 3), 0.4, 12) * scale
    ref, ref_abs = oracle.phi(X, with_abs=True)
    got = api.potential(_dev(X), mode="fp64").cpu().numpy()
    assert np.all(np.abs(got - ref) <= 1e-12 * ref_abs)


@pytest.mark.parametrize("far", [1e5, 1e7, 1e10, 1e14])
def test_fp64_one_far_point(far):
    """What the others feel does not depend on a point far away (the sweep's from about
    1e9 times the spacing on)."""
    X = inputs.uniform_cube(400, 400 ** (1 / 3), 0.4, 13)
    X[137] = far
    others = np.arange(400) != 137
    ref, ref_abs = oracle.phi(X, with_abs=True)
    got = api.potential(_dev(X), mode="fp64").cpu().numpy()
    assert np.all(np.abs(got - ref)[others] <= 1e-12 * ref_abs[others])
    F, S = oracle.forces(X, with_norm=True)
    got = api.forces(_dev(X), mode="fp64").cpu().numpy()
    assert np.all(np.abs(got - F).max(axis=1)[others] <= 1e-12 * S[others])


def test_fp64_pairs_closer_than_the_packed_points():
    """Points that differ in their last bits are distinct: solved, not refused."""
    X = inputs.uniform_cube(300, 300 ** (1 / 3), 0.4, 14)
    X[50] = X[51]
    X[50, 0] = np.nextafter(X[51, 0], 100.0)
    got = api.potential(_dev(X), mode="fp64").cpu().numpy()
    F = api.forces(_dev(X), mode="fp64").cpu().numpy()
    assert np.all(np.isfinite(got)) and np.all(np.isfinite(F))
    r = X[50, 0] - X[51, 0]
    assert min(abs(got[50]), abs(got[51])) > 0.1 * r ** -3
    X[50] = X[51]
    with pytest.raises(Exception) as e:
        api.potential(_dev(X), mode="fp64")
    assert getattr(e.value, "status", None) == -1
