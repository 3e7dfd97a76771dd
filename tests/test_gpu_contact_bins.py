"""GPU vs oracle: the soft-sphere contact kernels on either side of the occupancy rule and at the
edges of the binned kernel's runs, chunks and lists.

Forces and spins come from the common start-of-step state, as in test_gpu_soft_spheres.py: FP64
within 1e-11 and FP32 within 1e-5 of the largest.  Beds pressed far into each other run in FP64
only (an FP32 normal of nearly coincident centres loses the digits of their distance).
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


def _bed(name):
    if name == "2d-below":       # 4.9 particles per cell: the walk
        return W.packed_bed(n=(19, 23), fill_rows=23, n_particles=int(4.9 * 19 * 23))
    if name == "2d-above":       # 5.1: binned, short rows (several runs per block), ragged last block
        return W.packed_bed(n=(7, 61), fill_rows=61, n_particles=int(5.1 * 7 * 61))
    if name == "2d-periodic":    # runs over a whole row of three periodic cells
        return W.packed_bed(n=(3, 40), fill_rows=40, n_particles=1200).with_(bc=(P, P, P, P, P, P))
    if name == "2d-long-run":    # a row so sparse that its run is cut, above a crowded one
        w = W.packed_bed(n=(400, 6), fill_rows=2, n_particles=12800)
        x = (np.arange(0, 400, 3) + 0.5) * w.h
        pos = np.concatenate([w.pos, np.stack([x, np.full_like(x, 4.5 * w.h)], axis=1)])
        return w.with_(bc=(P, P, N, N, P, P), pos=pos, vel=np.concatenate([w.vel, np.zeros((len(x), 2))]))
    if name == "2d-thin-top":    # a crowded layer under rows of a few particles each
        w = W.packed_bed(n=(8, 60), fill_rows=24, n_particles=2400)
        y, x = np.meshgrid(np.arange(26, 60), np.arange(1, 8, 3), indexing="ij")
        pos = np.stack([(x.ravel() + 0.5) * w.h, (y.ravel() + 0.5) * w.h], axis=1)
        pos = np.concatenate([pos, pos + [0.18 * w.h, 0.0]])   # pairs in contact
        return w.with_(pos=np.concatenate([w.pos, pos]), vel=np.concatenate([w.vel, np.zeros_like(pos)]))
    if name == "3d-thin-top":    # the same in 3D: more runs than blocks that share them
        w = W.packed_bed(dim=3, n=(6, 7, 12), fill_rows=3, n_particles=int(7.5 * 504))
        z, y, x = np.meshgrid(np.arange(4, 12), np.arange(7), np.arange(0, 6, 2), indexing="ij")
        pos = (np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1) + 0.4) * w.h
        pos = np.concatenate([pos, pos + [0.0, 0.18 * w.h, 0.0]])
        return w.with_(pos=np.concatenate([w.pos, pos]), vel=np.concatenate([w.vel, np.zeros_like(pos)]))
    if name == "2d-pressed":     # more pairs than a list and more candidates than a chunk hold
        return W.packed_bed(n=(6, 10), fill_rows=5, n_particles=6 * 5 * 88, gap=0.3)
    if name == "3d-below":
        return W.packed_bed(dim=3, n=(7, 5, 9), fill_rows=9, n_particles=int(7.9 * 315))
    if name == "3d-above":
        return W.packed_bed(dim=3, n=(7, 5, 9), fill_rows=9, n_particles=int(8.1 * 315))
    assert name == "3d-pressed"
    return W.packed_bed(dim=3, n=(3, 4, 5), fill_rows=5, n_particles=60 * 250, gap=0.4).with_(
        bc=(P, P, P, P, N, N))


@pytest.mark.parametrize("name,storage", [
    ("2d-below", W.STORE_F32), ("2d-above", W.STORE_F32), ("2d-above", W.STORE_F64),
    ("2d-periodic", W.STORE_F32), ("2d-long-run", W.STORE_F32), ("2d-thin-top", W.STORE_F32), ("2d-pressed", W.STORE_F64),
    ("3d-below", W.STORE_F32), ("3d-above", W.STORE_F32), ("3d-thin-top", W.STORE_F32), ("3d-pressed", W.STORE_F64)])
@pytest.mark.parametrize("friction", [False, True])
def test_contact_kernels_against_oracle(name, storage, friction):
    from paper_1303_2653_gb300 import lbdps as L
    w = _bed(name)
    w = W.with_friction(w) if friction else w
    bed, ob = _pair(w, storage)
    bed.step(1)
    ob.step(1)
    tol = 1e-11 if storage == W.STORE_F64 else 1e-5
    fg, fo = bed.particle_diag(L.PDIAG_FC), ob.particle_diag(O.P_FC)
    assert np.abs(fg - fo).max() <= tol * np.abs(fo).max()
    np.testing.assert_array_equal(np.abs(fg).sum(axis=1) > 0, np.abs(fo).sum(axis=1) > 0)
    if friction:
        so = ob.spin()
        assert np.abs(bed.spin() - so).max() <= tol * np.abs(so).max()
    assert bed.check_guards() == 0
    bed.close()
