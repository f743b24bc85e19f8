"""The FP64 contraction with its columns in slabs (csrc/contract64.cu): whatever the
scratch, the same sums, and scratch that stays bounded as N grows (9 GB and a quarter)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,budget_mb", [(300, 20), (1100, 60), (1100, 120), (2500, 300)])
def test_slabs_agree_with_one_piece(n, budget_mb):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 22)
    Xd = torch.from_numpy(X).cuda()
    idx = inputs.sample_indices(n, 40, 3)
    _, ref_abs = oracle.phi(X, idx, with_abs=True)
    ctx = api.Context(0, budget_mb << 20)
    for call in (api.potential, api.forces):
        one = call(Xd, mode="fp64").cpu().numpy()
        got = call(Xd, mode="fp64", ctx=ctx).cpu().numpy()
        if got.ndim == 1:
            assert np.all(np.abs(got - one)[idx] <= 1e-13 * ref_abs)
        else:
            assert np.linalg.norm(got - one) <= 1e-13 * np.linalg.norm(one)
    assert (budget_mb << 20) * 0.3 < ctx.bytes_in_use() <= budget_mb << 20
    ctx.close()


def test_scratch_is_bounded():
    X = torch.from_numpy(inputs.uniform_cube(9000, 20.8, 0.3, 23)).cuda()
    ctx = api.Context(0)
    got = api.potential(X, mode="fp64", ctx=ctx).cpu().numpy()
    assert ctx.bytes_in_use() <= 12 << 30
    idx = inputs.sample_indices(9000, 8, 5)
    ref, ref_abs = oracle.phi(X.cpu().numpy(), idx, with_abs=True)
    assert np.all(np.abs(got[idx] - ref) <= 1e-12 * ref_abs)
    ctx.close()
