"""Pair terms of the FP32 triple sweep (csrc/exhaustive.cu), which serves potentials of
fewer than 1 280 particles: as accurate as the FP64 coordinates allow, at any offset, and
distinct points are distinct however close.

Bar: the one of the exhaustive tests, 3e-6 sum|phi|; with the one close pair, which makes
a single term of near-cancelling parts the whole sum, 3e-6 of the sum of the terms' parts
(oracle.phi_parts, the rounding scale of a term). The sweep's masked terms hold r^-6 of a
pair, in FP32: pairs down to 4e-7."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _phi(X):
    return api.potential(torch.from_numpy(np.ascontiguousarray(X)).cuda(), mode="fp32").cpu().numpy()


@pytest.mark.parametrize("n", [3, 33, 500])
@pytest.mark.parametrize("off", [0.0, 1e7, 1e10, 1e12])
def test_offset(n, off):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.4, 50 + n) + off
    ref, ref_abs = oracle.phi(X, with_abs=True)
    assert np.all(np.abs(_phi(X) - ref) <= 3e-6 * ref_abs)


def test_last_bit_apart():
    """Two points one FP64 step apart at 1e10 (1.9e-6)."""
    X = inputs.uniform_cube(300, 300 ** (1 / 3), 0.4, 14) + 1e10
    X[50] = X[51]
    X[50, 0] = np.nextafter(X[51, 0], 2e10)
    assert np.all(np.abs(_phi(X) - oracle.phi(X)) <= 3e-6 * oracle.phi_parts(X))
    X[50] = X[51]
    with pytest.raises(Exception) as e:
        _phi(X)
    assert getattr(e.value, "status", None) == -1
