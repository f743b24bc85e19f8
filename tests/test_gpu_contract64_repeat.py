"""FP64 potentials are sums of many contributions added in no fixed order: what each
addition rounds off is carried, so that repeated solves agree to the last bit of the result
(one unit, where the order of the carries themselves decides a tie), also where the terms
cancel to a small fraction of their magnitudes."""
import numpy as np
import pytest
import torch

from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [200, 700, 2049])
def test_repeated_solves_agree(n):
    X = torch.from_numpy(inputs.uniform_cube(n, n ** (1 / 3), 0.3, 600 + n)).cuda()
    first = api.potential(X, mode="fp64").cpu().numpy()
    for _ in range(6):
        again = api.potential(X, mode="fp64").cpu().numpy()
        assert np.all(np.abs(again - first) <= np.spacing(np.abs(first)))
