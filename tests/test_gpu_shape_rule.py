"""The launch shape of the reference block follows from what the domain is now, not from what it
has been."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def _shape(d):
    i = d.info()
    return tuple(i.tile), i.ctas_per_sm, i.nodes_per_thread


@pytest.mark.parametrize("storage,kind", [("fp32", "refined"), ("fp32", "far")])
def test_removing_the_last_block_restores_the_shape(lib, storage, kind):
    """1.2 M nodes: two nodes per thread alone, one beside another block."""
    from paper_1807_02284_gb300 import lbm
    dims = (128, 96, 96)
    d, fresh = lbm.Domain(dims, 0.01, storage=storage), lbm.Domain(dims, 0.01, storage=storage)
    alone = _shape(fresh)
    assert _shape(d) == alone
    for _ in range(2):
        if kind == "refined":
            b = d.add_scale_block((8.0, 8.0, 8.0), 0.5, (16, 16, 16))
        else:
            fb = synth.far_block(synth._empty_block(dims), 2.0, 16.0)
            b = d.add_scale_block(fb.origin, fb.h, fb.dims)
        assert _shape(d) != alone
        d.remove_scale_block(b)
        assert _shape(d) == alone
    d.set_walls((0, 0, 1, 1, 0, 0))
    assert _shape(d) != alone
    d.set_walls((0,) * 6)
    assert _shape(d) == alone
    d.close()
    fresh.close()


def test_steps_after_a_block_was_removed(lib):
    """A domain that had a refined and then a far-field block steps like one that never had."""
    import numpy as np
    from paper_1807_02284_gb300 import lbm
    from tests.helpers import f32, gpu_domain
    sc = synth.random_scene(dims=(36, 30, 28), seed=4, periodic=(False,) * 3, nu=0.01,
                            spheres=[(18.0, 15.0, 14.0, 4.0)])
    b = sc.blocks[0]
    d, ref = gpu_domain(sc), gpu_domain(sc)
    k = d.add_scale_block((4.0, 4.0, 4.0), 0.5, (12, 12, 12))
    d.step(3)
    d.remove_scale_block(k)
    fb = synth.far_block(b, 2.0, 8.0, seed=9)
    k = d.add_scale_block(fb.origin, fb.h, fb.dims)
    d.step(2)
    d.remove_scale_block(k)
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    for n in (5, 5, 20, 1):
        d.step(n)
        ref.step(n)
    for f in (lbm.LBM_FIELD_F, lbm.LBM_FIELD_U, lbm.LBM_FIELD_SCALAR):
        assert np.array_equal(d.read_field(f, lbm.LBM_F32), ref.read_field(f, lbm.LBM_F32))
    d.close()
    ref.close()


@pytest.mark.parametrize("dims,faces,obstacles,nodes", [
    ((176, 160, 152), False, False, 2), ((176, 160, 152), True, False, 2),
    ((176, 160, 152), False, True, 1), ((176, 160, 152), True, True, 1),
    ((256, 256, 256), True, True, 2), ((128, 96, 96), True, False, 1)])
def test_nodes_per_thread_with_walls(lib, dims, faces, obstacles, nodes):
    """Pairs from 2^20 nodes, with wall faces from 2^22, with obstacle-surface walls from 2^24."""
    from paper_1807_02284_gb300 import lbm
    d = lbm.Domain(dims, 0.01, storage="fp16")
    d.set_walls((0, 0, 0, 0, 1, 1) if faces else (0,) * 6, obstacles=obstacles)
    assert d.info().nodes_per_thread == nodes
    d.close()
