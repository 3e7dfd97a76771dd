"""The collision's thread mappings (along rows, along planes) at odd and small lattices: one step
against the oracle element by element, and the statistics summed in the same mapping."""
import os
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

from oracle import oracle as O                      # noqa: E402
from paper_1303_2653_gb300 import workloads as W    # noqa: E402
from test_gpu_parity import TOL, TOL_DERIVED, _pair, _rel   # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1303_2653_gb300 import build
    build.build_all()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# rows of a multiple of 32 and not; fewer cells than a warp and than a block; one row; a row longer
# than a block by one cell; enough blocks for 128 threads each; planes that end inside a warp; from
# (3, 13000) on, lattices large enough for threads along the plane
@pytest.mark.parametrize("n", [(3, 5), (31, 33), (32, 9), (33, 1), (129, 7), (250, 160), (5, 3, 4),
                               (32, 3, 5), (33, 31, 7), (3, 13000), (129, 310), (100, 9, 50),
                               (33, 31, 41)])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
def test_row_shapes(n, storage):
    from paper_1303_2653_gb300 import lbdps as L
    dim = len(n)
    # walls but for the last axis, which is periodic where it has the three cells that needs
    last = W.PERIODIC if n[-1] >= 3 else W.WALL
    bc = (W.WALL,) * (2 * dim - 2) + (last,) * 2 + (W.PERIODIC,) * (6 - 2 * dim)
    rng = np.random.default_rng(61)
    pos = (np.stack(np.meshgrid(*[np.arange(0, m, 2) for m in n], indexing="ij"), -1)
           .reshape(-1, dim) + rng.uniform(0.3, 0.7, size=dim))
    vel = rng.normal(0.0, 1e-2, size=pos.shape)
    w = W.Workload(name="rows", dim=dim, n=n, bc=bc, h=1.0, dt=1.0, d_p=0.3, rho_s=800.0, e=0.9,
                   pos=pos, vel=vel, rho_g=1.0, mu_g=0.01, body_accel=(1e-6, 0.0, 0.0),
                   u0=(0.0, 0.01, 0.0), cs_smag=0.1, storage=storage)
    bed, ob = _pair(w, storage)
    f0 = bed.populations() + rng.uniform(-1e-4, 1e-4, size=(bed.q, bed.ncell))
    bed.set_populations(f0)
    ob.set_populations(bed.populations())
    bed.step(1)
    ob.step(1)
    g = bed.fields(L.FIELD_RHO | L.FIELD_U | L.FIELD_FPG | L.FIELD_BETA)
    assert np.abs(g["rho"] - ob.field(O.F_RHO)).max() <= TOL[storage]
    assert _rel(g["u"], ob.field(O.F_U)) <= TOL[storage]
    assert _rel(g["fpg"], ob.field(O.F_FPG)) <= TOL_DERIVED[storage]
    assert _rel(g["beta"], ob.field(O.F_BETA)) <= TOL_DERIVED[storage]
    assert np.abs(bed.populations() - ob.populations()).max() <= TOL[storage]
    recs = L.Bed(w, storage=storage)       # monitored sums of a state equal lbdps_stats of it
    recs.set_populations(f0)
    got = recs.step_monitored(2)
    recs2 = L.Bed(w, storage=storage)
    recs2.set_populations(f0)
    for r in got:
        recs2.step(1)
        s = recs2.stats()
        assert r["mass"] == s["mass"] and np.array_equal(r["gas_momentum"], s["gas_momentum"])
    for b in (bed, recs, recs2):
        assert b.check_guards() == 0
        b.close()
