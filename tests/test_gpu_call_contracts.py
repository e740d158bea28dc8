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


@pytest.mark.parametrize("steps", [5, 9000])
def test_null_event_barrier_gives_up(fk, orc, steps):
    """The barrier between a step's parts waits for an arrival that never comes, gives
    up after 2 ms and reports it; no step is made or counted, later launches of the
    call make none, and the context stays usable."""
    cells, nv, nh = (12, 12, 12), 20, 60
    kw = dict(edge=4, precision=1, cap_v=32)
    b = fk.Batch([(*cells, 4.01)] * 3, [(nv, nh)] * 3, 3, test_stuck_wait_us=2000, **kw)
    b.set_barriers(0.7, 0.35, 800.0)
    before = [(b.state(r), b.records(r)) for r in range(3)]
    with pytest.raises(fk.KmcError) as e:
        b.run_null(steps, nv)
    assert e.value.code == fk.FKMC_ETIMEOUT
    for r in range(3):
        assert np.array_equal(b.state(r), before[r][0]) and np.array_equal(b.records(r), before[r][1])
        assert (b.info(r).null_steps, b.info(r).null_theta, b.info(r).hops) == (0, 0.0, 0)
    ok = fk.Batch([(*cells, 4.01)], [(nv, nh)], 3, **kw)
    ok.set_barriers(0.7, 0.35, 800.0)
    ok.run_null(30, nv)
    ref = orc.Lattice(cells, None, nv, nh, seed=3, edge=4)
    ref.set_rates(0.7, 0.35, 800.0, a_ang=4.01, cap_v=32, precision=1)
    ref.null_run(30, nv)
    assert np.array_equal(ok.records(), ref.records())
    assert ok.info().null_theta == ref.null_clock()["theta"]
