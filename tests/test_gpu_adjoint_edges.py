"""Adjoint at the extents where its tiles end: pass B covers 32 x 8 receivers of a plane and
marches in z, pass A walks the nodes of a plane, so rows just above a tile, the three-node
minimum, and open as well as periodic ends are compared with the FP64 oracle."""
import numpy as np
import pytest

import synth
from tests.test_gpu_adjoint import gpu_grad, oracle_grad, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,periodic", [((3, 3, 3), True), ((33, 9, 5), True),
                                           ((34, 3, 17), False), ((5, 17, 3), False),
                                           ((31, 8, 4), (True, False, True))])
def test_adjoint_at_tile_edges_matches_fp64_oracle(lib, dims, periodic):
    """Bound: FP32 against FP64 arithmetic over three steps, 1e-5 relative L2 (about 50 roundings
    of 6e-8 in every chain, summed in quadrature with their cancellations; the longer runs
    of the other adjoint tests hold 1e-3)."""
    per = (periodic,) * 3 if isinstance(periodic, bool) else periodic
    sc = synth.random_scene(dims=dims, seed=21, periodic=per, nu=0.01, amp=0.04)
    target = np.random.default_rng(2).random(sc.blocks[0].shape_zyx)
    L, g, _ = gpu_grad(sc, target, 3, 2)
    Lo, go, _ = oracle_grad(sc, target, 3)
    assert abs(L - Lo) <= 1e-5 * abs(Lo)
    assert rel(g, go.numpy()) <= 1e-5
