"""What the header promises of single calls: the rows that a read-out leaves alone,
the error that a device-side wait gives."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2004_09081_gb300 import fkmc
    fkmc.load()
    return fkmc


def test_rows_beyond_the_records_are_left_alone(fk):
    """A saved state whose replica row names more vacancies than it has records."""
    import torch
    nv, more = 20, 3
    b = fk.Batch([(12, 12, 12, 4.01)], [(nv, 40)], 8, edge=4, precision=1, cap_v=32)
    rec = b.records()
    n = fk.kmc_state_bytes(b.h)
    blob = torch.empty(n, dtype=torch.uint8).pin_memory()
    fk.kmc_download_state(b.h, blob.data_ptr(), n)
    row = blob[64:64 + 56].numpy().view(np.int64)  # window, steps, hops, hand-offs, clock, vacancies, H-
    assert row[5] == nv
    row[5] = nv + more
    fk.kmc_upload_state(b.h, blob.data_ptr(), n)
    assert b.info().n_vac == nv + more
    rows = np.full((nv + more, 6), -7, np.int64)
    total = ctypes.c_int64()
    fk._check(fk.load().kmc_read_records(b.h, 0, fk._ptr(rows), nv + more, ctypes.byref(total)))
    assert total.value == nv
    assert np.array_equal(rows[:nv], rec) and (rows[nv:] == -7).all()
