"""Monitored runs whose steps and reductions are launched in chunks: every record is the statistics
of the state that single steps reach, whatever the lengths of the calls and the parity they start on."""
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


# below the length that makes a chunk, at it, one and three steps over whole chunks, chunks from the
# other parity, a call shorter than that length once chunks are there, a single step
@pytest.mark.parametrize("calls", [(15, 16, 17), (17, 20, 5, 1, 6, 24), (1, 17, 3, 18)])
@pytest.mark.parametrize("storage", [W.STORE_F64, W.STORE_F32])
def test_records_of_chunks(calls, storage):
    from paper_1303_2653_gb300 import lbdps as L
    w = W.bubbling2d(nx=40, ny=80, n_particles=700, seed=11)     # inlet, outlet and walls
    bed, ref = L.Bed(w, storage=storage), L.Bed(w, storage=storage)
    for n in calls:
        recs = bed.step_monitored(n)
        assert len(recs) == n
        for got in recs:
            ref.step(1)
            want = ref.stats()
            assert got.keys() == want.keys()
            for key in want:
                # both sum the same values in the same order; not a number without diagnostics
                assert np.array_equal(got[key], want[key], equal_nan=True), (n, key)
    for a, b in zip(bed.particles(), ref.particles()):
        assert np.array_equal(a, b)
    assert bed.check_guards() == 0
    bed.close()
    ref.close()
