"""GPU vs oracle: the binned soft-sphere contacts of beds whose thin top spreads a block over many
runs of cells.

In 3D a run spans at most 111 cells and the blocks of a group of slots share its runs; beyond 3 runs
(2D, FP32; 8 in FP64) or 48 (3D) a block walks for the particles left.  Two steps, each from a
common start-of-step state: what a slot keeps from the step before must not pass for its force or
spin.  Bounds as in test_gpu_soft_spheres.py.
"""
import os
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

from oracle import oracle as O                      # noqa: E402
from paper_1303_2653_gb300 import workloads as W    # noqa: E402
from test_gpu_parity import _pair                   # noqa: E402

pytestmark = pytest.mark.gpu

P, N = W.PERIODIC, W.WALL


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1303_2653_gb300 import build
    build.build_all()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _top(w, rows, x):
    """w with a pair in contact in the cells x of every row of cells in rows (their y, or y and z)."""
    rows = np.asarray(rows).reshape(len(rows), -1)
    pos = np.column_stack([np.tile(x, len(rows)), np.repeat(rows, len(x), axis=0)]) + 0.4
    step = np.zeros(w.dim)
    step[0] = 0.18
    pos = np.concatenate([pos, pos + step]) * w.h
    vel = np.random.default_rng(len(pos)).normal(0.0, 0.05, size=pos.shape)
    return w.with_(pos=np.concatenate([w.pos, pos]), vel=np.concatenate([w.vel, vel]))


def _rows(w, first):
    """the rows of cells from level `first` of the vertical axis on"""
    if w.dim == 2:
        return np.arange(first, w.n[1])
    z, y = np.meshgrid(np.arange(first, w.n[2]), np.arange(w.n[1]), indexing="ij")
    return np.stack([y.ravel(), z.ravel()], axis=1)


def _check(w, storage):
    from paper_1303_2653_gb300 import lbdps as L
    bed, ob = _pair(w, storage)
    tol = 1e-11 if storage == W.STORE_F64 else 1e-5
    for step in range(2):
        if step:
            ob.set_populations(bed.populations())
            ob.set_particles(*bed.particles())
            if w.dem_mu > 0:
                ob.set_spin(bed.spin())
        bed.step(1)
        ob.step(1)
        fg, fo = bed.particle_diag(L.PDIAG_FC), ob.particle_diag(O.P_FC)
        assert np.abs(fg - fo).max() <= tol * np.abs(fo).max(), step
        if w.dem_mu > 0:
            so = ob.spin()
            assert np.abs(bed.spin() - so).max() <= tol * np.abs(so).max(), step
    assert bed.check_guards() == 0
    bed.close()


@pytest.mark.parametrize("nx,every", [(111, 8), (112, 1), (112, 3), (113, 2), (160, 1), (160, 8), (300, 1),
                                      (300, 2), (300, 24)])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
@pytest.mark.parametrize("friction", [False, True])
@pytest.mark.parametrize("bc", [(N,) * 6, (P, P, N, N, N, N)])
def test_rows_of_several_runs(nx, every, storage, friction, bc):
    # two crowded planes (9 particles per cell of the bed) under rows that hold a pair in every
    # `every`-th cell, so that 256 slots lie in one row, in two, or in nine and more
    w = W.packed_bed(dim=3, n=(nx, 4, 7), fill_rows=2, n_particles=9 * nx * 28)
    w = _top(w, _rows(w, 3), np.arange(0, nx, every)).with_(bc=bc)
    _check(W.with_friction(w) if friction else w, storage)


# pairs in a row of the top: runs of a block far beyond the limit, at it and just past it, below it
@pytest.mark.parametrize("dim,pairs", [(2, 1), (2, 8), (2, 14), (2, 16), (3, 1), (3, 2), (3, 3), (3, 9)])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
@pytest.mark.parametrize("friction", [False, True])
def test_thin_tops(dim, pairs, storage, friction):
    if dim == 2:
        w = W.packed_bed(n=(16, 60), fill_rows=24, n_particles=15 * 384, gap=0.8)
        w = _top(w, _rows(w, 25), np.arange(16)[::-1][:pairs])
    else:
        w = W.packed_bed(dim=3, n=(16, 6, 16), fill_rows=4, n_particles=39 * 384)
        w = _top(w, _rows(w, 5), np.arange(16)[::-1][:pairs])
    _check(W.with_friction(w) if friction else w, storage)


# either side of the rule that takes the binned kernel, and forms of it that only crowded rows reach
EDGES = [
    # 2D: 5.5 per cell in FP32, 5 in FP64; 66 and 22 per row; runs over a whole row of periodic cells
    ((64, 24), 8447, (N,) * 6), ((64, 24), 8448, (N,) * 6), ((64, 24), 7679, (N,) * 6), ((64, 24), 7680, (N,) * 6),
    ((11, 60), 3959, (N,) * 6), ((11, 60), 3960, (N,) * 6), ((4, 60), 1319, (N,) * 6), ((4, 60), 1320, (N,) * 6),
    ((3, 40), 120 * 23, (P,) * 6), ((13, 33), 429 * 7, (P, P, N, N, P, P)),
    # 3D: 8 per cell and, in FP32, 20 per row more, in FP64 16 per row at least
    ((24, 5, 9), 9539, (N,) * 6), ((24, 5, 9), 9540, (N,) * 6), ((24, 5, 9), 8639, (N,) * 6), ((24, 5, 9), 8640, (N,) * 6),
    ((3, 6, 7), 1847, (N,) * 6), ((3, 6, 7), 1848, (N,) * 6), ((1, 6, 7), 671, (N,) * 6), ((1, 6, 7), 672, (N,) * 6),
    ((3, 4, 5), 60 * 30, (P, P, P, P, N, N))]


@pytest.mark.parametrize("n,particles,bc", EDGES)
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
@pytest.mark.parametrize("friction", [False, True])
def test_either_side_of_the_rule(n, particles, bc, storage, friction):
    w = W.packed_bed(dim=len(n), n=n, fill_rows=n[-1], n_particles=particles, gap=0.7).with_(bc=bc)
    _check(W.with_friction(w) if friction else w, storage)


@pytest.mark.parametrize("friction", [False, True])
def test_long_sparse_rows_2d(friction):
    # a row so sparse that its run is cut, above crowded ones
    w = W.packed_bed(n=(400, 6), fill_rows=2, n_particles=13600, gap=0.8)
    w = _top(w, [4, 5], np.arange(0, 400, 3)).with_(bc=(P, P, N, N, P, P))
    _check(W.with_friction(w) if friction else w, W.STORE_F32)
