"""The FP32 bounds that settle most node triples of the tree potential: the
decisions have to be those of the FP64 rule, which the oracle restates, at
coordinate sizes, offsets and box shapes where FP32 bounds are loose (an offset
of many diameters, flat and needle-like sets). The tolerance is absolute: a
relative one is taken of potentials that the GPU sums in FP32 and the oracle in
FP64, which may decide a triple at the line by itself. Counts of prunes and visited
triples are whole numbers: equal."""
import numpy as np
import pytest

from oracle import tree as otree
from paper_1105_2769_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _set(shape, n=700):
    X = inputs.uniform_cube(n, n ** (1 / 3), 0.5, 91)
    if shape == "offset":
        return X + np.array([3e4, -2e4, 1e4])
    if shape == "small":
        return X * 2.0 ** -7
    if shape == "large":
        return X * 2.0 ** 9
    if shape == "flat":
        return X * np.array([4.0, 4.0, 0.25])
    if shape == "needle":
        return X * np.array([64.0, 1.0, 1.0])
    return X


@pytest.mark.parametrize("shape", ["cube", "offset", "small", "large", "flat", "needle"])
@pytest.mark.parametrize("tau_rel", [0.3, 30.0, 3000.0])
def test_decisions_are_those_of_the_fp64_rule(shape, tau_rel):
    import torch
    X = np.ascontiguousarray(_set(shape))
    Xd = torch.from_numpy(X).cuda()
    tau = tau_rel * float(np.median(np.abs(api.potential(Xd, mode="fp64").cpu().numpy())))
    _, st = api.potential(Xd, mode="tree_abs", eps=tau, stats=True)
    rst = otree.tree_potential(X, eps=0.0, alpha=0.0, tau=tau)[-1]
    assert (st["det_prunes"], st["node_triples_visited"]) == (rst["det_prunes"], rst["visited"])
