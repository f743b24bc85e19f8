"""Base cases at every leaf size a launch can meet (rows, columns and lanes of
leaves of 1 to 32 points), and the force-scale seed at ragged node sizes.

eps = 0 prunes nothing, so the solve is the exact sum: the bar is the FP32-bulk
one, 3e-6 sum|phi| for potentials and 3e-5 sum|grad phi| for forces."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf,n", [(2, 3), (2, 40), (3, 41), (5, 75), (8, 125), (11, 170),
                                    (14, 220), (16, 256), (17, 136), (18, 140), (20, 157),
                                    (21, 161), (24, 190), (25, 193), (28, 223), (29, 226),
                                    (32, 255), (32, 257), (32, 512)])
def test_leaf_sizes(leaf, n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 900 + n)
    ref, ref_abs = oracle.phi(X, with_abs=True)
    Xd = torch.from_numpy(X).cuda()
    cfg = api.tree_config(leaf_size=leaf, seed_levels=2)
    a = api.potential(Xd, eps=0.0, mode="tree", config=cfg).cpu().numpy()
    b = api.potential(Xd, eps=0.0, mode="tree", config=cfg).cpu().numpy()
    assert np.all(np.abs(a - ref) <= 3e-6 * ref_abs)
    # whatever the order of the base list: sums over lanes carry their rounding
    assert np.all(np.abs(a - b) <= 1e-12 * ref_abs)


@pytest.mark.parametrize("n,levels", [(3, 0), (33, 1), (70, 1), (257, 2), (300, 6), (601, 3)])
def test_force_scale_seed(n, levels):
    """A criterion that nothing meets (eps = 0) and one that all but the seed
    decides: the force error stays within eps S (a theorem at alpha = 0)."""
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 950 + n)
    F, S = oracle.forces(X, with_norm=True)
    Xd = torch.from_numpy(X).cuda()
    for eps in (0.0, 0.3):
        cfg = api.tree_config(leaf_size=8, seed_levels=levels)
        got = api.forces(Xd, mode="tree", eps=eps, config=cfg).cpu().numpy()
        assert np.all(np.abs(got - F).max(axis=1) <= (eps + 3e-5) * S)
