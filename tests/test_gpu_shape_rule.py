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
