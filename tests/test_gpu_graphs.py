"""Short runs of small blocks replayed from captured graphs: the same bits as single steps, over
re-initialisations, flag changes between runs, and under a caller's own stream capture."""
import numpy as np
import pytest

import synth
from tests.helpers import f32, gpu_domain

pytestmark = pytest.mark.gpu


def _scene():
    return synth.random_scene(dims=(20, 18, 16), seed=61, periodic=(False, True, False), nu=0.01,
                              spheres=[(10.0, 9.0, 8.0, 3.0)], inflow=(9, 8, 3.0, 0.08))


def _fields(d):
    from paper_1807_02284_gb300 import lbm
    return [d.read_field(f, lbm.LBM_F32) for f in (lbm.LBM_FIELD_F, lbm.LBM_FIELD_U, lbm.LBM_FIELD_SCALAR)]


@pytest.mark.parametrize("runs", [(7, 7, 7, 7), (3, 5, 3, 5, 3, 5), (17, 17, 17), (32, 9, 9, 9)])
def test_runs_equal_single_steps(lib, runs):
    sc = _scene()
    b = sc.blocks[0]
    a, c = gpu_domain(sc), gpu_domain(sc)
    other = (b.flags.copy())
    other[:, :, -2] |= synth.SCALAR_SRC
    for again in range(3):
        for d in (a, c):
            d.set_flags(other if again == 2 else b.flags)
            d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
        for n in runs:
            a.step(n)
            for _ in range(n):
                c.step(1)
        for x, y in zip(_fields(a), _fields(c)):
            assert np.array_equal(x, y)
        assert a.info().steps == sum(runs)
    a.close()
    c.close()


def test_step_under_the_callers_capture(lib):
    import torch
    from paper_1807_02284_gb300 import lbm
    sc = _scene()
    b = sc.blocks[0]
    st = torch.cuda.Stream()
    d = lbm.Domain(b.dims, sc.nu, periodic=sc.periodic, stream=st)
    d.set_flags(b.flags)
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    ref = gpu_domain(sc)
    for _ in range(3):
        d.step(4)
    d.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        g.capture_begin(capture_error_mode="thread_local")
        d.step(4)
        g.capture_end()
        for _ in range(2):
            g.replay()
    st.synchronize()
    ref.step(20)
    for x, y in zip(_fields(d), _fields(ref)):
        assert np.array_equal(x, y)
    d.close()
    ref.close()


@pytest.mark.parametrize("runs", [(4, 4, 4), (3, 1, 3, 3, 20, 20)])
def test_short_runs_on_a_stream_that_cannot_be_captured(lib, runs):
    """cudaStreamLegacy (handle 1): no graph can be captured on it, the steps are launched."""
    from paper_1807_02284_gb300 import lbm
    sc = _scene()
    b = sc.blocks[0]
    d = lbm.Domain(b.dims, sc.nu, periodic=sc.periodic, stream=1, torch_allocator=False)
    d.set_flags(b.flags)
    d.init_macro(f32(b.u0), rho=f32(b.rho0), c=f32(b.c0))
    ref = gpu_domain(sc)
    for n in runs:
        d.step(n)
    for _ in range(sum(runs)):
        ref.step(1)
    for x, y in zip(_fields(d), _fields(ref)):
        assert np.array_equal(x, y)
    d.close()
    ref.close()
