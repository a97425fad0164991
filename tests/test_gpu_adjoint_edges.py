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


@pytest.mark.parametrize("h", [1 / 3.0, 1 / 3.5])
def test_adjoint_of_blocks_with_more_than_two_levels_of_substeps(lib, h):
    """Refined blocks whose sub-steps reuse a time level within one reference step (three exact
    sub-steps, four with alignment): the scalar's departure velocity of each sub-step is its
    own.  Bound 1e-4 relative L2 (FP32 against FP64 over 2 reference steps, 6 to 8 sub-steps,
    with the mappings' atomic sums in any order)."""
    import torch

    from oracle import adjoint as oadj
    from paper_1807_02284_gb300 import lbm
    from tests.test_gpu_multiscale import gpu_multiscale
    sc = synth.multiscale(seed=2, sphere_seed=3, scale=0.125, flow_amp=0.03, nu=0.004)
    b1 = synth._empty_block((14, 13, 12), origin=(3.0, 4.0, 4.0), h=h)
    b1.u0, b1.rho0, b1.c0 = synth.smooth_field(b1, 11, amp=0.03, wavelength=8.0)
    sc.blocks = [sc.blocks[0], b1]
    target = np.zeros(sc.blocks[0].shape_zyx)
    dom = gpu_multiscale(sc)
    dom.set_tape(2)
    dom.step(2)
    c = dom.read_field(lbm.LBM_FIELD_SCALAR, lbm.LBM_F64)
    dc = torch.tensor(c, dtype=torch.float32, device="cuda")
    grads = [torch.empty(3 * b.flags.size, dtype=torch.float32, device="cuda") for b in sc.blocks]
    torch.cuda.synchronize()
    dom.adjoint_step(2, dc, grads[0])
    dom.adjoint_block_grad(1, grads[1])
    dom.sync()
    dom.close()
    _, go, _ = oadj.ms_loss_and_grad(sc, 2, target)
    for b, g, o in zip(sc.blocks, grads, go):
        assert rel(g.cpu().numpy().astype(np.float64).reshape(b.u0.shape), o.numpy()) <= 1e-4


def test_tape_buffers_are_reused_and_given_back(lib):
    """A second rollout takes the first one's tape buffers (no allocation), gives the same
    gradient, and the first step without a tape, or lbm_set_tape(0), gives them back."""
    import torch

    from paper_1807_02284_gb300 import lbm
    from tests.helpers import f32
    sc, _ = synth.adjoint_scene(n=14, seed=5, nu=0.01)
    b = sc.blocks[0]
    d = lbm.Domain(b.dims, sc.nu, periodic=sc.periodic)
    dc = torch.rand(b.flags.size, device="cuda")
    grads = [torch.empty(3 * b.flags.size, device="cuda") for _ in range(3)]
    torch.cuda.synchronize()

    def rollout(g):
        d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
        d.set_tape(2)
        d.step(5)
        d.adjoint_step(5, dc, g)
        d.sync()

    held = torch.cuda.memory_allocated
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    d.step(1)
    d.sync()
    bare = held()
    rollout(grads[0])
    with_tape = held()
    assert with_tape > bare
    rollout(grads[1])
    assert held() == with_tape
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    d.step(1)
    assert held() == bare
    rollout(grads[2])
    d.set_tape(0)
    assert held() == bare
    assert torch.equal(grads[0], grads[1]) and torch.equal(grads[0], grads[2])
    d.close()
