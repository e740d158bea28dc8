"""The null-event form's one launch for many steps where a thread holds two and
four vacancies and picks, and over several launches of its step log, against
the CPU oracle bit for bit."""
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


# 300 and 400 replicas whose vacancies do not fit one per thread on the GPU at once
@pytest.mark.parametrize("nrep,nv,n_frg", [(300, 400, 400), (400, 300, 250), (400, 300, 17)])
def test_several_vacancies_per_thread(fk, orc, nrep, nv, n_frg):
    cells, nf, nh = (8, 8, 8), (2, 2, 2), 200
    b = fk.Batch([(*cells, 4.01)] * nrep, [(nv, nh)] * nrep, 3, nfrag=nf, precision=1, tracer=True, cap_v=128)
    b.set_barriers(0.6, 0.4, 900.0)
    b.run_null(25, n_frg)
    for r in (0, 1, nrep // 2, nrep - 1):
        ref = orc.Lattice(cells, nf, nv, nh, seed=3, replica=r, tracer=True)
        ref.set_rates(0.6, 0.4, 900.0, a_ang=4.01, cap_v=128, precision=1)
        ref.null_run(25, n_frg)
        assert np.array_equal(b.state(r), ref.occupancy()), r
        assert np.array_equal(b.records(r), ref.records()), r
        assert np.array_equal(b.tracer_field(r), ref.tracer_field()), r
        assert b.info(r).null_theta == ref.null_clock()["theta"]
        assert b.info(r).hops == ref.counters()["hops"] > 0


def test_more_steps_than_one_log(fk, orc):
    cells, nf, nv, nh = (8, 8, 8), (2, 2, 2), 12, 60
    b = fk.Batch([(*cells, 4.01)], [(nv, nh)], 5, nfrag=nf, precision=0, cap_v=32)
    b.set_barriers(0.6, 0.4, 900.0)
    ref = orc.Lattice(cells, nf, nv, nh, seed=5)
    ref.set_rates(0.6, 0.4, 900.0, a_ang=4.01, cap_v=32, precision=0)
    for steps in (9000, 1):
        b.run_null(steps, 12)
        ref.null_run(steps, 12)
        assert np.array_equal(b.state(), ref.occupancy())
        assert np.array_equal(b.records(), ref.records())
        assert b.info().null_theta == ref.null_clock()["theta"]
