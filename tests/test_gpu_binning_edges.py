"""lbdps_bin_sort_noalloc at the edges of its tiles, digits and prefix tiles, against a NumPy
stable sort by (cell, id): equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1303_2653_gb300 import build
    build.build_all()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# one cell; the last lattice of one digit and the first of two; 4,095 and 4,096 cells (a prefix
# tile holds 4,096 counts, the list ncell + 1); digits of unequal width; particle counts around a
# tile of 1,024
@pytest.mark.parametrize("n", [(1, 1), (2, 1), (32, 32), (25, 41), (63, 65), (64, 64), (3, 5, 137)])
@pytest.mark.parametrize("count", [1, 1023, 1024, 1025, 40000])
def test_binning_edges(n, count):
    import torch
    from paper_1303_2653_gb300 import lbdps as L
    rng = np.random.default_rng(41 + count)
    P = rng.uniform(0, 1, size=(count, len(n))) * np.array(n, dtype=float)
    P[: count // 3] = P[0]                       # a crowded cell beside the others
    q = np.minimum(np.floor(P).astype(np.int64), np.array(n) - 1)
    cell = q[:, 0] + n[0] * (q[:, 1] + (n[1] * q[:, 2] if len(n) == 3 else 0))
    ncell = int(np.prod(n))
    dev = [torch.from_numpy(np.ascontiguousarray(P[:, a])).cuda() for a in range(len(n))]
    start = torch.full((ncell + 1,), -1, dtype=torch.int32, device="cuda")
    order = torch.full((count,), -1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(2):                           # the scratch keeps what the first call left
        L.bin_sort_noalloc(len(n), n, [t.data_ptr() for t in dev], start.data_ptr(), order.data_ptr(),
                           count, stream)
    np.testing.assert_array_equal(start.cpu().numpy(),
                                  np.r_[0, np.cumsum(np.bincount(cell, minlength=ncell))])
    np.testing.assert_array_equal(order.cpu().numpy(), np.argsort(cell, kind="stable"))


# one scan tile; the last tile count of one scan per scatter block and beyond 256 tiles; the largest
# lattice in small tiles and the first in large ones
@pytest.mark.parametrize("n", [(7, 9), (64, 64), (1024, 1027), (2048, 2047), (2048, 2048)])
def test_handle_sort_across_tile_counts(n):
    from paper_1303_2653_gb300 import lbdps as L
    from paper_1303_2653_gb300 import workloads as W
    rng = np.random.default_rng(43)
    blocks = (n[0] // 2) * (n[1] // 2)           # 2 x 2 cells, at most one particle each
    cells = rng.choice(blocks, size=min(3000, blocks), replace=False)
    pos = np.stack([2 * (cells % (n[0] // 2)), 2 * (cells // (n[0] // 2))], axis=1) + \
        rng.uniform(0.3, 1.3, size=(len(cells), 2)) * 0.7
    w = W.Workload(name="tiles", dim=2, n=n, bc=(W.PERIODIC,) * 6, h=1.0, dt=1.0, d_p=0.2, rho_s=800.0,
                   e=0.9, pos=pos, vel=rng.normal(0.0, 0.2, size=pos.shape), rho_g=1.0, mu_g=0.1)
    bed = L.Bed(w, storage=W.STORE_F32)
    for _ in range(3):
        bed.step(1)
        P, _ = bed.particles()
        q = np.floor(P).astype(np.int64)
        cell = q[:, 0] + n[0] * q[:, 1]
        np.testing.assert_array_equal(bed.particle_diag(L.PDIAG_ORDER), np.lexsort((np.arange(len(cell)), cell)))
        np.testing.assert_array_equal(bed.particle_diag(L.PDIAG_CELL), cell)
    assert bed.check_guards() == 0
    bed.close()
