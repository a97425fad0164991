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


def _runtime_calls(fn):
    """CUDA runtime calls by name made in fn()."""
    from torch.profiler import ProfilerActivity, profile

    def counts(f):
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
        return {e.key: e.count for e in prof.key_averages()}

    for _ in range(3):                    # a process's first profile can come back empty
        if counts(lambda: torch.ones(4, device="cuda").add_(1)).get("cudaLaunchKernel"):
            return counts(fn)
    pytest.skip("no CUDA activity records")


def test_batch_under_the_callers_capture(lib):
    """A batch first called while the caller captures its stream is captured as launches, replays
    to the same bits, and leaves no plan without a graph: the next calls replay graphs."""
    from paper_1807_02284_gb300 import lbm
    st = torch.cuda.Stream()
    a, b = _members(5, [st]), _members(5, [st])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="thread_local")
        lbm.step_batch(a, 4)
        g.capture_end()
        for _ in range(2):
            g.replay()
    st.synchronize()
    for d in b:
        d.step(8)
    _same(a, b)
    lbm.step_batch(a, 4)                  # (a plan is captured here at the latest)
    calls = _runtime_calls(lambda: lbm.step_batch(a, 4))
    assert calls.get("cudaGraphLaunch", 0) == 1, calls
    for d in b:
        d.step(8)
    _same(a, b)
    for d in a + b:
        d.close()


def test_batch_on_a_stream_that_cannot_be_captured(lib):
    """Members on cudaStreamLegacy (handle 1): their plan is a graph all the same."""
    from paper_1807_02284_gb300 import lbm
    scenes = synth.batch(count=3, seed=41, lo=8, hi=20, nu=2e-3)
    a, b = [], [gpu_domain(s) for s in scenes]
    for s in scenes:
        k = s.blocks[0]
        d = lbm.Domain(k.dims, s.nu, periodic=s.periodic, adaptive=s.adaptive, c_src=s.c_src,
                       stream=1, torch_allocator=False)
        d.set_flags(k.flags)
        d.init_macro(f32(k.u0), rho=f32(k.rho0), c=f32(k.c0))
        a.append(d)
    lbm.step_batch(a, 4)
    calls = _runtime_calls(lambda: lbm.step_batch(a, 4))
    assert calls.get("cudaGraphLaunch", 0) == 1, calls
    r = lbm.step_batch_reduce(a, 3)
    for d in b:
        d.step(11)
    _same(a, b)
    for x, d in zip(r, b):
        assert abs(x[0] - d.reduce()[0]) <= 1e-6 * x[0]
    for d in a + b:
        d.close()


@pytest.mark.parametrize("streams", [1, 3])
@pytest.mark.parametrize("steps", [17, 20])
def test_more_members_than_branches_with_diagnostics(lib, streams, steps):
    """40 members share 32 branches; a whole 16-step graph and its rest: the states of single
    steps bit for bit, the diagnostics those of lbm_step_reduce (the same records, summed in FP64:
    1e-13 of the sums' sizes), for both forms of the call and from both levels."""
    from paper_1807_02284_gb300 import lbm
    a, b = (_members(40, [torch.cuda.Stream() for _ in range(streams)], lo=6, hi=14) for _ in range(2))
    out = torch.zeros((40, 5), dtype=torch.float64, pin_memory=True)
    for k in range(3):
        if k == 1:
            a[0].wait_results(lbm.step_batch_reduce_async(a, steps, out))
            r = out.numpy()
        else:
            r = lbm.step_batch_reduce(a, steps)
        for d, x in zip(b, r):
            y = d.step_reduce(steps)
            n = d.n_nodes()
            assert np.abs(x - y).max() <= 1e-13 * n
        _same(a, b)
    for d in a + b:
        d.close()
