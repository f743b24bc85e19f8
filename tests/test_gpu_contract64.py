"""The FP64 contraction in exact fp16 products (csrc/contract64.cu) against the
FP64 oracle, at the edges of its tiles (128), blocks (256 columns, 512 above
N = 2 048) and batches, and on clustered and tied sets.

Bars: the FP64 ones of the exhaustive tests, 1e-12 |Phi| for potentials and
1e-12 sum|grad phi| for forces."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


@pytest.mark.parametrize("n", [192, 257, 320, 383, 384, 385, 512, 513, 769, 2048, 2049, 2561])
def test_potential_at_tile_edges(n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 600 + n)
    idx = np.unique(np.concatenate([inputs.sample_indices(n, 40, n), [0, n - 1]]))
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    got = api.potential(_dev(X), mode="fp64").cpu().numpy()[idx]
    assert np.all(np.abs(got - ref) <= 1e-12 * np.minimum(np.abs(ref), ref_abs))


@pytest.mark.parametrize("n", [96, 127, 128, 129, 255, 256, 257, 385, 700])
def test_forces_at_tile_edges(n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 700 + n)
    F, S = oracle.forces(X, with_norm=True)
    assert np.all(np.abs(api.forces(_dev(X), mode="fp64").cpu().numpy() - F).max(axis=1) <= 1e-12 * S)


def test_clustered_and_tied_sets():
    g = np.arange(9, dtype=np.float64)
    lattice = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) * 0.75
    for X in (lattice, inputs.gaussian_mixture(900, 3, 6.0, 0.1, 2.0, 0.01, 11),
              inputs.uniform_cube(900, 1.2, 0.01, 12)):
        ref, ref_abs = oracle.phi(X, with_abs=True)
        got = api.potential(_dev(X), mode="fp64").cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-12 * ref_abs)
        F, S = oracle.forces(X, with_norm=True)
        assert np.all(np.abs(api.forces(_dev(X), mode="fp64").cpu().numpy() - F).max(axis=1)
                      <= 1e-12 * S)


def test_batches_agree_with_one_piece():
    """Scratch for a few tiles at a time, and for none (the sweep)."""
    X = inputs.uniform_cube(1100, 10.3, 0.3, 21)
    Xd = _dev(X)
    one = api.potential(Xd, mode="fp64").cpu().numpy()
    for budget in (260 << 20, 2 << 20):
        ctx = api.Context(0, budget)
        got = api.potential(Xd, mode="fp64", ctx=ctx).cpu().numpy()
        np.testing.assert_allclose(got, one, rtol=1e-12)
        ctx.close()
