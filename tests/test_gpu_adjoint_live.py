"""The reverse sweep belongs to the recorded run: what the caller writes into the live state
afterwards (the next frame's inflow records, node boxes), or on a checkpoint's boundary, does
not reach the departure velocities of the steps before it."""
import numpy as np
import pytest
import torch

import synth
from oracle import adjoint as oadj
from oracle import grid
from tests.helpers import f32
from tests.test_gpu_adjoint import rel

pytestmark = pytest.mark.gpu


def _scene(scale=1.0, periodic=(True, True, True)):
    """Random flow and scalar with an inflow disk whose nodes are not scalar sources."""
    sc, target = synth.adjoint_scene(n=12, seed=11, nu=0.01, amp=0.05)
    sc.periodic = periodic
    b = sc.blocks[0]
    b.c0 = np.random.default_rng(9).random(b.c0.shape)
    synth.inflow_disk(b, (6, 6), 3.0, 0.12 * scale, rng=np.random.default_rng(3), noise=0.5,
                      scalar=False)
    return sc, target


def _record(sc, every, stream=None, storage="fp32"):
    from paper_1807_02284_gb300 import lbm
    b = sc.blocks[0]
    d = lbm.Domain(b.dims, sc.nu, periodic=sc.periodic, stream=stream, storage=storage)
    d.set_flags(b.flags)
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    d.set_tape(every)
    return d


def _grad(d, steps, target):
    n = d.n_nodes()
    dc = torch.tensor(target.reshape(-1) - 0.5, dtype=torch.float32, device="cuda")
    g = torch.empty(3 * n, device="cuda")
    torch.cuda.synchronize()
    d.adjoint_step(steps, dc, g)
    d.sync()
    return g.cpu().numpy()


@pytest.mark.parametrize("how", ["records", "batch", "box"])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("steps,every", [(1, 3), (6, 3), (7, 3)])
def test_state_written_after_the_run_leaves_the_gradient(lib, how, storage, steps, every):
    from paper_1807_02284_gb300 import lbm
    if how == "box" and storage == "fp16":
        pytest.skip("node boxes need FP32 storage")
    sc, target = _scene()
    other, _ = _scene(-1.0)
    st = torch.cuda.Stream()
    out = []
    for write in (False, True):
        d, e = _record(sc, every, st, storage), _record(sc, every, st, storage)
        for x in (d, e):
            x.step(steps)
        if write and how == "records":
            d.set_inflow(synth.inflow_records(other.blocks[0]))
        elif write and how == "batch":
            lbm.set_inflow_batch([e, d], [synth.inflow_records(other.blocks[0])] * 2)
        elif write:
            lo, hi = (0, 0, 0), tuple(v - 1 for v in sc.blocks[0].dims)
            buf = torch.empty((d.box_bytes(0, lo, hi) + 3) // 4, device="cuda")
            torch.cuda.synchronize()
            d.pack_box(0, lbm.LBM_LEVEL_CURRENT, lo, hi, buf)
            d.sync()
            buf.mul_(-0.5)
            torch.cuda.synchronize()
            d.unpack_box(0, lbm.LBM_LEVEL_CURRENT, lo, hi, buf)
        out.append(_grad(d, steps, target))
        d.close()
        e.close()
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))


@pytest.mark.parametrize("periodic", [(True, True, True), (False, False, False)])
def test_records_on_a_checkpoint_boundary(lib, periodic):
    """New inflow velocities after step 3 of 6 with a checkpoint every 3: the first segment keeps
    its own velocities, the second starts from the new ones (the change itself passed through, as
    every stored state).  Bound 1e-5 relative L2: FP32 against FP64 over six steps."""
    sc, target = _scene(periodic=periodic)
    other, _ = _scene(-1.0, periodic)
    b = sc.blocks[0]
    d = _record(sc, 3)
    d.step(3)
    d.set_inflow(synth.inflow_records(other.blocks[0]))
    d.step(3)
    g = _grad(d, 6, target)
    d.close()
    p = grid.Params(nu=sc.nu, periodic=sc.periodic, adaptive=sc.adaptive)
    start = [f32(a).astype(np.float64) for a in (b.u0, b.rho0, b.c0)]
    u0 = torch.tensor(start[0], requires_grad=True)
    with torch.no_grad():
        mid = oadj.forward(torch.tensor(start[0]), start[1], start[2], b.flags, p, 3)
        inflow = torch.as_tensor((b.flags & synth.INFLOW) != 0)
        new = torch.tensor(f32(other.blocks[0].u0).astype(np.float64))
        u = torch.where(inflow[None], new, mid.u)
    end = oadj.forward(u0, start[1], start[2], b.flags, p, 6, restart={3: (mid.f, u, mid.c)})
    (end.c * torch.tensor(f32(target.reshape(end.c.shape) - 0.5).astype(np.float64))).sum().backward()
    assert rel(g.astype(np.float64).reshape(b.u0.shape), u0.grad.numpy()) <= 1e-5
