"""Plans of the batched calls: several members per branch, whole graphs and their rest, calls that
fail, and calls under the caller's own stream capture."""
import numpy as np
import pytest
import torch

import synth
from tests.helpers import f32, gpu_domain

pytestmark = pytest.mark.gpu


def _members(count, streams, seed=40, lo=8, hi=20):
    from paper_1807_02284_gb300 import lbm
    out = []
    for i, s in enumerate(synth.batch(count=count, seed=seed, lo=lo, hi=hi, nu=2e-3)):
        b = s.blocks[0]
        d = lbm.Domain(b.dims, s.nu, periodic=s.periodic, adaptive=s.adaptive, c_src=s.c_src,
                       stream=streams[i % len(streams)])
        d.set_flags(b.flags)
        d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
        out.append(d)
    return out


def _fields(d):
    from paper_1807_02284_gb300 import lbm
    return [d.read_field(f, lbm.LBM_F32) for f in (lbm.LBM_FIELD_F, lbm.LBM_FIELD_U, lbm.LBM_FIELD_SCALAR)]


def _same(xs, ys):
    for x, y in zip(xs, ys):
        for a, b in zip(_fields(x), _fields(y)):
            assert np.array_equal(a, b)


def test_a_call_without_its_plan_leaves_the_members(lib, monkeypatch):
    """20 steps take a graph of 16 and one of 4 with diagnostics buffers: when those cannot be
    allocated, no member has moved, and the same call works once there is memory."""
    from paper_1807_02284_gb300 import lbm
    streams = [torch.cuda.Stream() for _ in range(2)]
    a, b = _members(4, streams), _members(4, streams)
    real = torch.cuda.caching_allocator_alloc

    def none(*_):
        raise RuntimeError("no memory")

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", none)
    with pytest.raises(lbm.LBMError) as err:
        lbm.step_batch_reduce(a, 20)
    assert err.value.status == lbm.LBM_ERR_OOM
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", real)
    assert all(d.info().steps == 0 for d in a)
    _same(a, b)
    lbm.step_batch_reduce(a, 20)
    for d in b:
        d.step(20)
    assert all(d.info().steps == 20 for d in a)
    _same(a, b)
    for d in a + b:
        d.close()
