"""Device buffers of the adjoint: a failed allocation leaves the tape as it was, so that the
same call works once there is memory again."""
import numpy as np
import pytest
import torch

import synth
from tests.helpers import f32
from tests.test_gpu_adjoint import rel
from tests.test_gpu_multiscale import gpu_multiscale

pytestmark = pytest.mark.gpu


class Allocations:
    """Counts the library's device allocations and what they hold; number `fail_at` fails (the
    caller's allocator raises, the library gets NULL)."""

    def __init__(self, monkeypatch):
        self.count, self.fail_at, self.live = 0, -1, {}
        real, real_free = torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

        def alloc(nbytes, device=None, stream=None):
            self.count += 1
            if self.count - 1 == self.fail_at:
                raise RuntimeError("no memory")
            p = real(nbytes, device, stream)
            self.live[p] = nbytes
            return p

        def free(p):
            self.live.pop(p, None)         # (None: taken before this test)
            real_free(p)

        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
        monkeypatch.setattr(torch.cuda, "caching_allocator_delete", free)

    def held(self):
        return sum(self.live.values())


def _scene(blocks):
    if blocks == 1:
        sc, _ = synth.adjoint_scene(n=12, seed=5, nu=0.01)
        sc.periodic = (False, False, True)
        return sc
    sc = synth.multiscale(seed=2, sphere_seed=3, scale=0.125, flow_amp=0.03, nu=0.004)
    sc.blocks = sc.blocks[:2]
    return sc


def _domain(sc):
    from paper_1807_02284_gb300 import lbm
    if len(sc.blocks) > 1:
        return gpu_multiscale(sc)
    b = sc.blocks[0]
    d = lbm.Domain(b.dims, sc.nu, periodic=sc.periodic)
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    return d


@pytest.mark.parametrize("blocks", [1, 2])
def test_reverse_sweep_after_a_failed_allocation(lib, monkeypatch, blocks):
    """Every allocation of lbm_adjoint_step in turn: OOM, then the same call gives the
    gradient.  Bound 1e-5: one block repeats its bits; the mappings' atomic sums of at most 16
    corners come in any order, 2^-24 each, over three steps."""
    from paper_1807_02284_gb300 import lbm
    sc = _scene(blocks)
    mem = Allocations(monkeypatch)
    n = sc.blocks[0].flags.size
    dc = torch.rand(n, device="cuda")
    ref, fail = None, -1
    while True:
        d = _domain(sc)
        d.set_tape(2)
        d.step(3)
        g = torch.full((3 * n,), 7.0, device="cuda")
        torch.cuda.synchronize()
        mem.count, mem.fail_at = 0, fail
        failed = False
        try:
            d.adjoint_step(3, dc, g)
        except lbm.LBMError as err:
            assert err.status == lbm.LBM_ERR_OOM
            failed = True
            mem.fail_at = -1
            d.adjoint_step(3, dc, g)
        d.sync()
        mem.fail_at = -1
        d.close()
        g = g.cpu().numpy().astype(np.float64)
        if ref is None:
            ref, total = g, mem.count
            assert total > 0 and not failed
        else:
            assert failed and rel(g, ref) <= 1e-5, fail
        fail += 1
        if fail == total:
            break


@pytest.mark.parametrize("blocks", [1, 2])
def test_a_released_tape_holds_no_memory(lib, monkeypatch, blocks):
    """lbm_init_macro releases the tape and with it all of its memory, whatever comes next (a step,
    a batched step, another domain's rollout): nothing but the domain's own is held then."""
    sc = _scene(blocks)
    held = Allocations(monkeypatch).held
    n = sc.blocks[0].flags.size
    dc, g = torch.rand(n, device="cuda"), torch.empty(3 * n, device="cuda")
    torch.cuda.synchronize()
    d = _domain(sc)
    d.step(1)
    d.sync()
    bare = held()
    for every in (2, 3, 1):
        for i, b in enumerate(sc.blocks):
            d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0), block=i)
        assert held() == bare
        d.set_tape(every)
        d.step(5)
        assert held() > bare
        d.adjoint_step(5, dc, g)
        d.sync()
    d.init_macro(f32(sc.blocks[0].u0))
    assert held() == bare
    d.close()


@pytest.mark.parametrize("blocks", [1, 2])
def test_gradients_do_not_depend_on_what_the_memory_held(lib, blocks):
    """Checkpoint intervals changed from rollout to rollout on one domain, its buffers taken from
    memory full of NaN: the gradient of a fresh domain each time.  Bound: as above."""
    sc = _scene(blocks)
    n = sc.blocks[0].flags.size
    dc = torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def rollout(d, every):
        for i, b in enumerate(sc.blocks):
            d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0), block=i)
        dirty = [torch.full((1 << 22,), float("nan"), device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        del dirty
        g = torch.empty(3 * n, device="cuda")
        d.set_tape(every)
        d.step(5)
        d.adjoint_step(5, dc, g)
        d.sync()
        return g.cpu().numpy().astype(np.float64)

    d = _domain(sc)
    for every in (2, 5, 1, 3, 2):
        fresh = _domain(sc)
        ref = rollout(fresh, every)
        fresh.close()
        assert np.isfinite(ref).all() and rel(rollout(d, every), ref) <= 1e-5, every
    d.close()
