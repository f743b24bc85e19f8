"""FP64 potentials and forces beside a tight group of many points: its pairs are near pairs
(csrc/near.cu), so that its rows do not cost the others digits of their fixed-point terms.

Bars: 1e-12 sum|phi| and 1e-12 sum|grad phi|, the FP64 ones of the exhaustive tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,members,size", [(2049, 10, 1e-4), (8000, 30, 1e-3)])
def test_others_keep_their_digits(n, members, size):
    rng = np.random.default_rng(8)
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.5, 77)
    X = np.concatenate([X, X[17] + 0.3 + rng.normal(size=(members, 3)) * size])
    X = np.ascontiguousarray(X[rng.permutation(n + members)])
    Xd = torch.from_numpy(X).cuda()
    idx = inputs.sample_indices(n + members, 150, 9)
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    got = api.potential(Xd, mode="fp64").cpu().numpy()[idx]
    assert np.all(np.abs(got - ref) <= 1e-12 * ref_abs)
    F, S = oracle.forces(X, idx[:60], with_norm=True)
    got = api.forces(Xd, mode="fp64").cpu().numpy()[idx[:60]]
    assert np.all(np.abs(got - F).max(axis=1) <= 1e-12 * S)
