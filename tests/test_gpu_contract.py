"""The tensor-core contraction behind the FP32 exhaustive modes (csrc/contract.cu)
against the FP64 oracle, at the edges of its tiles (128 rows, 256 columns),
windows (64) and blocks (256), with scratch that forces slabs and batches, and
on sets whose closest pairs dwarf the rest or tie (the pairs that are summed
term by term).

Bars: the FP32 ones of the exhaustive tests, 3e-6 sum|phi| for potentials and
3e-5 sum|grad phi| for gradients."""
import numpy as np
import pytest
import torch

import oracle
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


@pytest.mark.parametrize("n", [96, 127, 128, 129, 255, 256, 257, 320, 385, 513])
def test_gradients_at_tile_edges(n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 400 + n)
    g = inputs.random_weights(n, 401 + n)
    F, S = oracle.forces(X, with_norm=True)
    assert np.all(np.abs(api.forces(_dev(X), mode="fp32").cpu().numpy() - F).max(axis=1) <= 3e-5 * S)
    G, S = oracle.vjp(X, g, with_norm=True)
    got = api.potential_vjp(_dev(X), _dev(g), mode="fp32").cpu().numpy()
    assert np.all(np.abs(got - G).max(axis=1) <= 3e-5 * S)


@pytest.mark.parametrize("n", [1280, 1281, 1535, 1537, 2305])
def test_potential_at_tile_edges(n):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.3, 500 + n)
    idx = inputs.sample_indices(n, 48, n)
    idx = np.unique(np.concatenate([idx, [0, n - 1]]))
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    got = api.potential(_dev(X), mode="fp32").cpu().numpy()[idx]
    assert np.all(np.abs(got - ref) <= 3e-6 * ref_abs)


def test_slabs_and_batches_agree_with_one_piece():
    """100 MB of scratch: six slabs of columns, and batches of tiles for the VJP."""
    X = inputs.gaussian_mixture(1500, 1, 11.3, 0.5, 3.0, 0.05, 7)
    g = inputs.random_weights(1500, 8)
    Xd, gd = _dev(X), _dev(g)
    _, ab = oracle.phi(X, np.arange(0, 1500, 50), with_abs=True)
    small = api.Context(0, 100 << 20)
    a = api.potential(Xd, mode="fp32").cpu().numpy()
    b = api.potential(Xd, mode="fp32", ctx=small).cpu().numpy()
    assert small.bytes_in_use() > 40 << 20  # the contraction ran
    assert np.all(np.abs(a - b)[::50] <= 3e-6 * ab)
    for f in (lambda c: api.forces(Xd, mode="fp32", ctx=c),
              lambda c: api.potential_vjp(Xd, gd, mode="fp32", ctx=c)):
        one, many = f(None).cpu().numpy(), f(small).cpu().numpy()
        assert np.linalg.norm(one - many) <= 3e-6 * np.linalg.norm(one)
    tiny = api.Context(0, 1 << 20)  # no room: the triple sweep
    c = api.forces(Xd, mode="fp32", ctx=tiny).cpu().numpy()
    one = api.forces(Xd, mode="fp32").cpu().numpy()
    assert np.linalg.norm(one - c) <= 3e-6 * np.linalg.norm(c)
    small.close()
    tiny.close()


@pytest.mark.parametrize("ratio", [10.0, 300.0])
def test_isolated_dimers(ratio):
    """Pairs `ratio` times closer than their spacing: their terms must not set the
    scale that the others are cut against."""
    n = 1400
    rng = np.random.default_rng(3)
    c = inputs.uniform_cube(n // 2, (n // 2) ** (1 / 3), 0.5, 5)
    d = rng.normal(size=c.shape)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    X = np.concatenate([c, c + d * (0.55 / ratio)])[rng.permutation(n)]
    idx = inputs.sample_indices(n, 40, 6)
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    got = api.potential(_dev(X), mode="fp32").cpu().numpy()[idx]
    assert np.all(np.abs(got - ref) <= 3e-6 * ref_abs)
    F, S = oracle.forces(X, with_norm=True)
    assert np.all(np.abs(api.forces(_dev(X), mode="fp32").cpu().numpy() - F).max(axis=1) <= 3e-5 * S)


def test_invalid_points_are_reported():
    X = inputs.uniform_cube(1300, 11.0, 0.3, 9)
    for bad in ("nan", "same"):
        Y = X.copy()
        if bad == "nan":
            Y[700, 2] = np.nan
        else:
            Y[1299] = Y[3]
        with pytest.raises(Exception) as e:
            api.potential(_dev(Y), mode="fp32")
        assert getattr(e.value, "status", None) == -1
    good = api.potential(_dev(X), mode="fp32").cpu().numpy()
    assert np.all(np.isfinite(good))


def test_lattice_ties():
    """Six nearest neighbours at one distance: all of them are near pairs."""
    g = np.arange(11, dtype=np.float64)
    X = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3) * 0.75
    idx = inputs.sample_indices(len(X), 32, 2)
    ref, ref_abs = oracle.phi(X, idx, with_abs=True)
    got = api.potential(_dev(X), mode="fp32").cpu().numpy()[idx]
    assert np.all(np.abs(got - ref) <= 3e-6 * ref_abs)
    F, S = oracle.forces(X, with_norm=True)
    assert np.all(np.abs(api.forces(_dev(X), mode="fp32").cpu().numpy() - F).max(axis=1) <= 3e-5 * S)
