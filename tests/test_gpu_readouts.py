"""Read-outs expanded on the device: occupancy bytes and record rows against the
oracle's, for row lengths around the 16 sites of a word, one fragment holding
many records, and fewer rows asked for than there are records."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [(1, 2, 3), (15, 4, 5), (16, 4, 4), (17, 6, 4), (33, 5, 7), (64, 8, 8)])
def test_state_and_records(orc, cells):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2004_09081_gb300 import fkmc as fk
    n = 3 * int(np.prod(cells))
    nv, nh = max(1, n // 16), n // 8
    b = fk.Batch([(8, 8, 8, 4.01), (*cells, 4.01)], [(9, 0), (nv, nh)], 6, edge=4, precision=0, cap_v=256)
    ref = orc.Lattice(cells, tuple(b.info(1).nfrag), nv, nh, seed=6, replica=1)
    assert np.array_equal(b.state(1), ref.occupancy())
    rec = b.records(1)
    assert np.array_equal(rec, ref.records())
    some = np.full((nv, 6), -7, np.int64)
    total = ctypes.c_int64()
    k = nv // 2
    fk._check(fk.load().kmc_read_records(b.h, 1, fk._ptr(some), k, ctypes.byref(total)))
    assert total.value == nv and np.array_equal(some[:k], rec[:k]) and (some[k:] == -7).all()
