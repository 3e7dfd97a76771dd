"""GPU vs oracle: the binned soft-sphere contacts of a 3D bed whose rows are cut into several runs
while the blocks of a group of slots share those runs.

A run spans at most 111 cells.  Two steps, each from a common start-of-step state: what a slot keeps
from the step before must not pass for its force or spin.  Bounds as in test_gpu_soft_spheres.py.
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


def _bed(nx, every, bc):
    """Two crowded planes (9 particles per cell of the bed) under rows that hold a pair in contact in
    every `every`-th cell, so that 256 slots lie in one row, in two, or in nine and more."""
    n = (nx, 4, 7)
    w = W.packed_bed(dim=3, n=n, fill_rows=2, n_particles=9 * nx * 28)
    z, y, x = np.meshgrid(np.arange(3, 7), np.arange(4), np.arange(0, nx, every), indexing="ij")
    pos = (np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1) + 0.4) * w.h
    pos = np.concatenate([pos, pos + [0.18 * w.h, 0.0, 0.0]])
    vel = np.random.default_rng(nx).normal(0.0, 0.05, size=pos.shape)
    return w.with_(bc=bc, pos=np.concatenate([w.pos, pos]), vel=np.concatenate([w.vel, vel]))


@pytest.mark.parametrize("nx,every", [(111, 8), (112, 1), (112, 3), (113, 2), (160, 1), (160, 8), (300, 1),
                                      (300, 2), (300, 24)])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
@pytest.mark.parametrize("friction", [False, True])
@pytest.mark.parametrize("bc", [(N,) * 6, (P, P, N, N, N, N)])
def test_rows_of_several_runs(nx, every, storage, friction, bc):
    from paper_1303_2653_gb300 import lbdps as L
    w = _bed(nx, every, bc)
    w = W.with_friction(w) if friction else w
    assert len(w.pos) >= 8 * nx * 28   # the binned kernel
    bed, ob = _pair(w, storage)
    tol = 1e-11 if storage == W.STORE_F64 else 1e-5
    for step in range(2):
        if step:
            ob.set_populations(bed.populations())
            ob.set_particles(*bed.particles())
            if friction:
                ob.set_spin(bed.spin())
        bed.step(1)
        ob.step(1)
        fg, fo = bed.particle_diag(L.PDIAG_FC), ob.particle_diag(O.P_FC)
        assert np.abs(fg - fo).max() <= tol * np.abs(fo).max(), step
        if friction:
            so = ob.spin()
            assert np.abs(bed.spin() - so).max() <= tol * np.abs(so).max(), step
    assert bed.check_guards() == 0
    bed.close()
