"""Launch shapes of the collide-stream step: CTAs of one row walk a plane's nodes in x-fastest
order and run on over the ends of rows; every shape computes the same values."""
import numpy as np
import pytest

import synth
from tests.helpers import gpu_domain

pytestmark = pytest.mark.gpu


def _state(monkeypatch, tile, sc, storage, walls):
    from paper_1807_02284_gb300 import lbm
    if tile:
        monkeypatch.setenv("LBM_TILE", tile)
    else:
        monkeypatch.delenv("LBM_TILE", raising=False)
    d = gpu_domain(sc, storage)
    if walls:
        d.set_walls((0, 0, 1, 1, 0, 0), obstacles=True)
    d.step(3)
    diag = d.step_reduce(1)
    out = [d.read_field(f, lbm.LBM_F32) for f in (lbm.LBM_FIELD_F, lbm.LBM_FIELD_U, lbm.LBM_FIELD_SCALAR)]
    d.close()
    return out, diag


@pytest.mark.parametrize("dims", [(1, 1, 1), (2, 3, 2), (31, 5, 3), (33, 4, 3), (34, 7, 5), (65, 9, 4),
                                  (96, 3, 2), (130, 6, 3)])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("walls", [False, True])
def test_one_row_ctas_equal_tiles(lib, monkeypatch, dims, storage, walls):
    """The chosen shape and one-row CTAs of both kernels against 32 x 8 tiles: equal bits; the
    diagnostics to FP32 rounding of their partial sums (2^-24 times the 256 terms of a CTA)."""
    spheres = [(dims[0] / 2, dims[1] / 2, dims[2] / 2, 1.2)] if min(dims) > 2 else ()
    sc = synth.random_scene(dims=dims, seed=31, periodic=(False, False, True), nu=0.01, spheres=spheres)
    ref, dref = _state(monkeypatch, "32,8,3", sc, storage, walls)
    for tile in ("", "32,1,3", "64,1,4", "128,1,4", "256,1,3", "64,1,20", "128,1,21", "256,1,22"):
        got, d = _state(monkeypatch, tile, sc, storage, walls)
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), tile
        assert np.abs(d - dref).max() <= 256 * 2.0 ** -24 * np.abs(dref).max()


@pytest.mark.parametrize("dims", [(36, 30, 28), (34, 9, 11)])
def test_pairs_with_ghost_and_obstacle_nodes_equal_single_nodes(lib, monkeypatch, dims):
    """A block with obstacles inside a far-field block (its outer nodes are scale-boundary
    ones): two nodes per thread give the bits of one node per thread in every block."""
    from paper_1807_02284_gb300 import lbm
    from tests.test_gpu_multiscale import gpu_multiscale
    sc = synth.random_scene(dims=dims, seed=4, periodic=(False,) * 3, nu=0.01, amp=0.04)
    rng = np.random.default_rng(8)
    solid = rng.random(sc.blocks[0].flags.shape) < 0.05
    solid[:3] = solid[-3:] = False
    solid[:, :3] = solid[:, -3:] = False
    solid[:, :, :3] = solid[:, :, -3:] = False
    sc.blocks[0].flags[solid] = synth.SOLID
    sc.blocks.append(synth.far_block(sc.blocks[0], 2.0, 8.0, seed=9))
    out = []
    for tile in ("128,1,4", "64,2,20", "128,1,20"):
        monkeypatch.setenv("LBM_TILE", tile)
        dom = gpu_multiscale(sc)
        dom.step(5)
        out.append([dom.read_field(lbm.LBM_FIELD_F, lbm.LBM_F64, block=b) for b in (0, 1)])
        dom.close()
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], o))


def _terms(d):
    """Per-node terms of the five diagnostics of the stored state in 64 bits (5, nodes): rho - 1,
    j, |j|^2 / (2 rho), over the nodes that count."""
    from paper_1807_02284_gb300 import lbm
    from oracle.cmr import C
    f = d.read_field(lbm.LBM_FIELD_F, lbm.LBM_F64).reshape(27, -1)
    fl = d.read_field(lbm.LBM_FIELD_FLAGS, lbm.LBM_U8).reshape(-1)
    keep = (fl & (synth.SOLID | synth.GHOST)) == 0
    rho = f.sum(0)
    j = np.einsum("qn,qa->an", f, np.asarray(C, dtype=np.float64))
    return np.concatenate([(rho - 1.0)[None], j, (0.5 * (j * j).sum(0) / rho)[None]])[:, keep], keep.sum()


@pytest.mark.parametrize("dims", [(31, 5, 3), (34, 7, 5), (96, 3, 2), (130, 16, 12)])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_every_diagnostic_within_its_own_terms(lib, monkeypatch, dims, storage):
    """lbm_step_reduce of every shape, bounce-back obstacle and inflow included: each of mass,
    momentum and energy against the 64-bit sums of the stored state, bounded by its own terms.  A
    term is taken before the collision, which conserves it to the rounding of some 40 operations on
    moments of at most a tenth (2^-22 of the node's weight of 1); a CTA's sum takes at most 256
    additions (256 * 2^-24 of the terms' magnitudes); FP16 storage is rounded after the sums are
    taken, 2^-11 of deviations of at most a tenth of each weight."""
    from paper_1807_02284_gb300 import lbm
    spheres = [(dims[0] / 2, dims[1] / 2, dims[2] / 2, 1.2)] if min(dims) > 2 else ()
    sc = synth.random_scene(dims=dims, seed=33, periodic=(False, False, True), nu=0.01, spheres=spheres)
    for tile in ("", "32,8,3", "64,1,4", "128,1,4", "64,2,20", "128,1,21"):
        if tile:
            monkeypatch.setenv("LBM_TILE", tile)
        else:
            monkeypatch.delenv("LBM_TILE", raising=False)
        d = gpu_domain(sc, storage)
        d.step(2)
        diag = d.step_reduce(1)
        t, n = _terms(d)
        d.close()
        per_node = 2.0 ** -22 if storage == "fp32" else 2.0 ** -22 + 0.1 * 2.0 ** -11
        u = np.sqrt((t[1:4] ** 2).sum(0)).max()
        exact, size = t.sum(1), np.abs(t).sum(1)
        exact[0] += n
        node = np.array([1, 1, 1, 1, 2 * u]) * per_node * n
        assert np.all(np.abs(diag - exact) <= 256 * 2.0 ** -24 * size + node), (tile, diag, exact)
