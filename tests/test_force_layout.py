"""The particles' force on the gas in 3D: kept per occupied cell below a particle per cell and per
cell from there on, so that a bed never holds more of it than the smaller of the two."""
import os
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

from paper_1303_2653_gb300 import workloads as W    # noqa: E402

P, N = W.PERIODIC, W.WALL


@pytest.mark.parametrize("storage,particle", [(W.STORE_F64, 280), (W.STORE_F32, 196)])
def test_crowded_bed_holds_the_force_per_cell(storage, particle):
    # bytes of a soft sphere in a bed of more particles than cells: P, v, in-cell offset, id and cell
    # in two lists, P, v and offset staged, key, slot, id of the slot, partner and wall, contact force
    from paper_1303_2653_gb300 import build, lbdps as L
    build.build_all()
    s = 8 if storage == W.STORE_F64 else 4
    assert particle == 2 * (24 + 6 * s + 8) + (24 + 6 * s) + (4 + 8 + 4 + 4 + 4) + 3 * s
    w = W.packed_bed(dim=3, n=(16, 16, 16), fill_rows=16, n_particles=8 * 4096)
    few = w.with_(pos=w.pos[:4 * 4096], vel=w.vel[:4 * 4096])
    grown = L.memory_estimate(w, storage) - L.memory_estimate(few, storage)
    assert abs(grown / (4 * 4096) - particle) < 1   # buffers are rounded up to 256 bytes


@pytest.mark.gpu
@pytest.mark.parametrize("particles", [1, 119, 120, 121, 240])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
def test_force_on_either_side_of_a_particle_per_cell(particles, storage):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from test_gpu_parity import _compare_step, _pair
    n = (4, 5, 6)   # one sphere in each quarter point of a cell's diagonal, cells in random order
    rng = np.random.default_rng(particles)
    cells = rng.permutation(120)
    at = np.concatenate([cells, cells])[:particles]
    off = np.repeat([0.25, 0.75], 120)[:particles, None]
    pos = np.stack([at % 4, at // 4 % 5, at // 20], axis=1) + off
    w = W.Workload(name="force", dim=3, n=n, bc=(N, N, N, N, P, P), h=1.0, dt=1.0, d_p=0.3, rho_s=800.0,
                   e=0.9, pos=pos, vel=rng.normal(0.0, 1e-2, size=pos.shape), rho_g=1.0, mu_g=0.01,
                   body_accel=(0.0, 0.0, 1e-6), u0=(0.0, 0.0, 0.01), cs_smag=0.1, storage=storage)
    bed, ob = _pair(w, storage)
    for step in range(2):
        if step:
            ob.set_populations(bed.populations())
            ob.set_particles(*bed.particles())
        _compare_step(bed, ob, storage)
    assert bed.check_guards() == 0
    bed.close()
