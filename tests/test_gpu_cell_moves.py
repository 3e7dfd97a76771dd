"""Moves across cell faces: the new cell and in-cell offset that the drag derives without FP64
equal those of the FP64 position, for velocities that end a step next to a cell face, on one,
beyond the neighbouring cell, at the faces of the lattice, at rest and subnormal."""
import os
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))

from paper_1303_2653_gb300 import workloads as W    # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1303_2653_gb300 import build
    build.build_all()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _state(dim, n):
    """A particle in every other cell of every other row, with a velocity from the list."""
    eps = [0.0, 1e-9, 1e-7, 5e-7, 3e-6, 5e-6, 1e-4, 0.2]
    ends = [s * e + base for base in (0.0, 1.0) for e in eps for s in (-1, 1)] + [0.5, 1.7, -0.6]
    rng = np.random.default_rng(51)
    grids = np.meshgrid(*[np.arange(0, m, 2) for m in n], indexing="ij")
    cell = np.stack([g.ravel() for g in grids], axis=1).astype(float)
    off = rng.uniform(0.25, 0.75, size=cell.shape)
    # velocities that carry the offset to one of the end points (relative to the cell)
    vel = rng.choice(np.array(ends), size=cell.shape) - off
    still = rng.uniform(size=cell.shape)
    vel[still < 0.1] = 0.0
    vel[(still >= 0.1) & (still < 0.2)] = 1e-40
    return cell + off, vel.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("dim,n,bc", [
    (2, (18, 22), (W.WALL, W.WALL, W.PERIODIC, W.PERIODIC, W.PERIODIC, W.PERIODIC)),
    (3, (10, 12, 14), (W.WALL,) * 4 + (W.PERIODIC,) * 2)])
@pytest.mark.parametrize("storage", [W.STORE_F32, W.STORE_F64])
def test_cell_and_offset_after_a_move(dim, n, bc, storage):
    from paper_1303_2653_gb300 import lbdps as L
    pos, vel = _state(dim, n)
    # heavy particles and a gas at rest: the drag hardly moves them off their end points
    w = W.Workload(name="moves", dim=dim, n=n, bc=bc, h=1.0, dt=1.0, d_p=0.2, rho_s=1e9, e=0.9,
                   pos=pos, vel=np.zeros_like(pos), rho_g=1.0, mu_g=0.1, storage=storage)
    bed = L.Bed(w, storage=storage)
    bed.set_particles(pos, vel)
    bed.step(1)
    saved = bed.save()
    P, v = bed.particles()
    assert np.all((P >= 0) & (P < np.array(n)))
    q = np.floor(P).astype(np.int64)
    lin = q[:, 0] + n[0] * (q[:, 1] + (n[1] * q[:, 2] if dim == 3 else 0))
    np.testing.assert_array_equal(bed.particle_diag(L.PDIAG_CELL), lin)
    # off the faces the move is one exact FP64 sum (no contacts: the particles start apart; the
    # pairs that meet change velocity only after the move)
    moved = pos + vel
    inner = np.all((moved > 0.01) & (moved < np.array(n) - 0.01), axis=1)
    assert inner.mean() > 0.4
    assert np.abs(P[inner] - moved[inner]).max() <= 1e-6
    # a bed with this state whose offsets come from the FP64 positions takes the same next step (the
    # checkpoint keeps the populations' bits, which their exported full values round)
    other = L.Bed(w, storage=storage)
    other.load(saved)
    other.set_particles(P, v)
    bed.step(1)
    other.step(1)
    for a, b in zip(bed.particles(), other.particles()):
        np.testing.assert_array_equal(a, b)
    for b in (bed, other):
        assert b.health() & 2 == 0
        b.close()
