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
