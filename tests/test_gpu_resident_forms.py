"""The resident window kernels (one CTA or a thread-block cluster per replica,
both arithmetic forms) against the CPU oracle where their parts change over:
row scans of every box shape, fragment lists that overflow and refill, first
draws made ahead and during a visit, the two forms of the clock, and the plain
form's draws in several chunks.  Everything is compared bit for bit."""
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


def pair(fk, orc, cells, nf, nv, nh, seed, prec, T=900.0, Ez=2e7, cap=64, n_tau=1.0, ctas=0, tracer=True, kernel=None):
    b = fk.Batch([(*cells, 4.01)], [(nv, nh)], seed, nfrag=nf, precision=prec, tracer=tracer, cap_v=cap, n_tau=n_tau,
                 cluster_ctas=ctas)
    b.set_barriers(0.6, 0.4, T, field_z=Ez)
    ref = orc.Lattice(cells, nf, nv, nh, seed=seed, tracer=tracer)
    ref.set_rates(0.6, 0.4, T, Ez=Ez, a_ang=4.01, cap_v=cap, n_tau=n_tau, precision=prec)
    assert b.info().kernel == (kernel if kernel is not None else 2 if ctas else 1)
    return b, ref


def check(b, ref, calls):
    for w in calls:
        b.run(w)
        ref.run(w)
        assert np.array_equal(b.state(), ref.occupancy())
        assert np.array_equal(b.records(), ref.records())
        assert np.array_equal(b.tracer_field(), ref.tracer_field())
        c = ref.counters()
        assert (b.info().hops, b.info().handoffs) == (c["hops"], c["handoffs"])
    assert ref.counters()["hops"] > 100


# extents 2 and 3; 5 and 6 (rows across word boundaries); 8; 9; 11 to 13 (more cells per
# lane than a mask holds); 18 and 40 (pieces of rows)
@pytest.mark.parametrize("cells,nf", [((8, 10, 8), (4, 4, 4)), ((20, 22, 24), (4, 4, 4)), ((32, 16, 32), (4, 2, 4)),
                                      ((36, 18, 18), (4, 2, 2)), ((24, 26, 22), (2, 2, 2)), ((36, 12, 12), (2, 2, 2)),
                                      ((40, 6, 8), (1, 2, 2))])
@pytest.mark.parametrize("prec", [0, 1])
def test_row_scans_of_every_box(fk, orc, prec, cells, nf):
    n = 3 * int(np.prod(cells))
    nv = min(6 * int(np.prod(nf)), n // 20)
    check(*pair(fk, orc, cells, nf, nv, n // 12, 5, prec), (25, 1, 30))


@pytest.mark.parametrize("ctas", [0, 2, 4])
@pytest.mark.parametrize("prec", [0, 1])
def test_lists_overflow_and_refill(fk, orc, prec, ctas):
    """Eight vacancies per fragment on average: a fragment's list (8) fills, gives
    way to the row scan and comes back; one CTA and 2 and 4 slabs."""
    check(*pair(fk, orc, (10, 12, 16), (2, 2, 4), 128, 400, 3, prec, ctas=ctas), (20, 20, 20))


@pytest.mark.parametrize("prec", [0, 1])
def test_long_windows_leave_the_clock_estimates(fk, orc, prec):
    """60 vacancies in one fragment at n_tau 64: thousands of events per visit.
    The mixed clock meets ratios below its last place and goes on in FP64; the
    plain clock fills its log many times and meets sums within 2^-10 of the
    window."""
    b, ref = pair(fk, orc, (8, 8, 8), (1, 1, 1), 60, 0, 7, prec, Ez=0.0, n_tau=64.0)
    check(b, ref, (6, 6))
    assert ref.counters()["hops"] > 30000


@pytest.mark.parametrize("ctas", [0, 2])
@pytest.mark.parametrize("prec", [0, 1])
def test_many_windows_in_one_call(fk, orc, prec, ctas):
    """More than two chunks of the plain form's draws (64 windows each), and
    colour orders of more than two blocks of 64 windows."""
    check(*pair(fk, orc, (8, 8, 12), (2, 2, 4), 20, 90, 11, prec, ctas=ctas, n_tau=0.5), (150, 3, 200))


VV = [(2, 0.343), (4, 0.235), (6, 0.200)]
FE = [(1, -0.709), (5, -0.199), (9, -0.022)]


# 16^3 cells fit one CTA; forced slabs; dense fragments (lists overflow, more than two chunks)
@pytest.mark.parametrize("cells,nf,nv,ctas", [((16, 16, 16), (4, 4, 4), 30, 0), ((16, 16, 24), (4, 4, 6), 40, 4),
                                              ((10, 11, 12), (2, 2, 2), 90, 0), ((10, 11, 16), (2, 2, 4), 140, 2)])
def test_site_energies_in_the_resident_kernels(fk, orc, cells, nf, nv, ctas):
    """Vacancy-vacancy and dopant shells: rates from the energy field, which every
    exchange moves, and marks on all fragments within the shells' reach."""
    b = fk.Batch([(*cells, 3.905)], [(nv, 60, 20)], 9, nfrag=nf, precision=0, tracer=True, cap_v=64,
                 cluster_ctas=ctas)
    b.set_site_energy(VV, FE)
    b.set_barriers(0.6, 0.4, 900.0, field_z=1e7)
    ref = orc.Lattice(cells, nf, nv, 60, seed=9, n_Fe=20, tracer=True)
    ref.set_site_energy(vv=VV, fe=FE)
    ref.set_rates(0.6, 0.4, 900.0, Ez=1e7, cap_v=64)
    assert b.info().kernel == (2 if ctas else 1)
    check(b, ref, (25, 1, 30))
    assert np.array_equal(b.site_field(), [ref.site_energy(s) for s in range(ref.nsite)])


def test_many_small_fragments_with_short_lists(fk, orc):
    """4,096 fragments of 2 x 2 x 2 cells in one layer: too many for lists of eight
    entries in one CTA's shared memory, and one layer cannot be cut into slabs."""
    cells, nf = (128, 128, 2), (64, 64, 1)
    check(*pair(fk, orc, cells, nf, 900, 4000, 3, 1, cap=16), (12, 1))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("cells,nf,nv,kernel", [
    ((32, 32, 32), (8, 8, 8), 511, 1),    # below 64 vacancies per phase: one CTA
    ((32, 32, 32), (8, 8, 8), 512, 2),    # four visits per warp and phase: a cluster
    ((24, 24, 24), (12, 12, 12), 40, 2),  # 216 fragments per phase
    ((64, 64, 2), (32, 32, 1), 2600, 0),  # over the line of both forms: the phase passes
])
def test_dense_replicas_change_kernels(fk, orc, prec, cells, nf, nv, kernel):
    check(*pair(fk, orc, cells, nf, nv, 500, 5, prec, kernel=kernel), (8, 1, 40))
