"""Paths that no other comparison with the oracle takes: the colour-phase passes in
the plain form where the replica would fit the resident kernels, with and without
site energies; the two-CTA slabs of kmc_opts.cluster_top; the mixed clock beyond
its integer form; rates that underflow to zero; long vacancy lists; the multigrid's
four-plane kernels where the planes do not divide by four; tables that grow within
a call."""
import numpy as np
import pytest

from oracle import poisson as ps

pytestmark = pytest.mark.gpu

VV = [(2, 0.343), (4, 0.235), (6, 0.200), (8, 0.180), (10, 0.023)]
FE = [(1, -0.709), (5, -0.199), (9, -0.022)]


@pytest.fixture(scope="module")
def fk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2004_09081_gb300 import fkmc
    fkmc.load()
    return fkmc


def check(b, ref, calls, tracer=True, hops=100, field=False):
    for w in calls:
        b.run(w)
        ref.run(w)
        assert np.array_equal(b.state(), ref.occupancy())
        assert np.array_equal(b.records(), ref.records())
        if tracer:
            assert np.array_equal(b.tracer_field(), ref.tracer_field())
        c = ref.counters()
        assert (b.info().hops, b.info().handoffs, b.info().window) == (c["hops"], c["handoffs"], c["window"])
    if field:
        assert np.array_equal(b.site_field(), [ref.site_energy(s) for s in range(ref.nsite)])
    assert ref.counters()["hops"] > hops


# one fragment per colour; several and uneven ones; one fragment of 60 vacancies, 15 chunks of events
@pytest.mark.parametrize("cells,nf,nv,nh", [((8, 8, 8), (2, 2, 2), 15, 51), ((8, 8, 12), (2, 2, 4), 30, 150),
                                            ((10, 12, 9), (2, 4, 2), 25, 60), ((8, 8, 8), (1, 1, 1), 60, 200)])
@pytest.mark.parametrize("small", [-1, 1])
def test_plain_passes(fk, orc, small, cells, nf, nv, nh):
    """The general pass, and the grouped one (one or two vacancies, four or two per warp)
    beside it."""
    b = fk.Batch([(*cells, 4.01)], [(nv, nh)], 3, nfrag=nf, precision=0, tracer=True, cap_v=64, schedule=1,
                 small_pass=small)
    b.set_barriers(0.6, 0.4, 900.0, field_z=2e7)
    ref = orc.Lattice(cells, nf, nv, nh, seed=3, tracer=True)
    ref.set_rates(0.6, 0.4, 900.0, Ez=2e7, a_ang=4.01, cap_v=64)
    assert b.info().kernel == 0
    check(b, ref, (60, 1, 60))


# the smallest edge the shells allow; uneven fragments; more vacancies than two chunks hold
@pytest.mark.parametrize("cells,nf,nv,nh", [((16, 16, 16), (4, 4, 4), 150, 0), ((16, 18, 20), (4, 4, 4), 60, 300),
                                            ((10, 11, 12), (2, 2, 2), 90, 60)])
def test_site_energy_passes(fk, orc, cells, nf, nv, nh):
    b = fk.Batch([(*cells, 3.905)], [(nv, nh, 30)], 9, nfrag=nf, precision=0, tracer=True, cap_v=64, schedule=1)
    b.set_site_energy(VV, FE)
    b.set_barriers(0.6, 0.3, 900.0, field_z=1e7)
    ref = orc.Lattice(cells, nf, nv, nh, seed=9, n_Fe=30, tracer=True)
    ref.set_site_energy(vv=VV, fe=FE)
    ref.set_rates(0.6, 0.3, 900.0, Ez=1e7, cap_v=64)
    assert b.info().kernel == 0
    check(b, ref, (25, 1, 30), field=True, hops=50)


@pytest.mark.parametrize("shells", [False, True])
def test_frozen_potential_passes(fk, orc, shells):
    cells, nf = (16, 16, 16), (4, 4, 4)
    b = fk.Batch([(*cells, 4.01)], [(60, 80)], 7, nfrag=nf, precision=0, tracer=True, cap_v=64, schedule=1)
    ref = orc.Lattice(cells, nf, 60, 80, seed=7, tracer=True)
    if shells:
        b.set_site_energy(VV, [])
        ref.set_site_energy(vv=VV)
    b.set_barriers(0.7, 0.5, 900.0, field_z=1e7)
    b.set_electrostatics(eps_r=100.0, refresh_windows=0)
    u = np.random.default_rng(1).integers(-1500, 1500, 3 * 16 ** 3).astype(np.int32)
    g = np.full((3, 8), -180, np.int32)
    b.write_potential_energy(u, g)
    ref.set_elec(u, g)
    ref.set_rates(0.7, 0.5, 900.0, Ez=1e7, a_ang=4.01, cap_v=64)
    assert b.info().kernel == 0
    check(b, ref, (40, 40), field=True)


def test_two_cta_slabs(fk, orc):
    """The largest replicas of the largest shared-memory class on two CTAs, half of the
    fragment layers each: 64 fragments and fewer than 64 vacancies per phase, so that
    the rule for many visits leaves them alone."""
    cells, comps, Ts = [(48, 48, 48), (48, 40, 56)], [(400, 9000), (380, 4000)], [700.0, 900.0]
    b = fk.Batch([(*c, 4.01) for c in cells], comps, 13, nfrag=(8, 8, 8), precision=1, cap_v=32, cluster_top=2,
                 tracer=True)
    b.set_barriers(0.6, 0.4, Ts)
    for calls in (20, 1, 40):
        b.run(calls)
    for r, (c, (nv, nh), T) in enumerate(zip(cells, comps, Ts)):
        assert (b.info(r).kernel, b.info(r).ctas) == (1, 2)
        ref = orc.Lattice(c, (8, 8, 8), nv, nh, seed=13, replica=r, tracer=True)
        ref.set_rates(0.6, 0.4, T, a_ang=4.01, cap_v=32, precision=1)
        ref.run(61)
        assert b.info(r).hops == ref.counters()["hops"] > 100
        assert np.array_equal(b.state(r), ref.occupancy()) and np.array_equal(b.records(r), ref.records())
        assert np.array_equal(b.tracer_field(r), ref.tracer_field())


def variate(orc, seed, window, event):
    """-ln u of an event of fragment 0 in the mixed form, as the oracle draws it."""
    x = orc.philox4x64([0, window, event // 2, 0], [seed, 3])  # purpose 3: hops
    return orc.neglog32(x[2 * (event & 1)])


# 60 vacancies: resident kernel and general pass; 4 vacancies: the same, and the two
# one-thread-per-fragment passes.  (seed, window, event) of a variate small enough
@pytest.mark.parametrize("nv,seed,window,event", [(60, 23, 7, 692), (60, 11, 6, 2908), (4, 887, 14, 67),
                                                  (4, 2871, 49, 126)])
@pytest.mark.parametrize("sched,small,lane", [(2, -1, 0), (1, -1, 0), (1, 1, 1), (1, 1, 2)])
def test_mixed_clock_beyond_its_integer_form(fk, orc, nv, seed, window, event, sched, small, lane):
    """A window of n_tau 64 is 105 units of 1/k32max (exponent 6), whose last place is
    2^-46: a ratio of an exponent below 6 - 29 turns the clock to FP64 for the rest of
    the visit.  All vacancies lie in one fragment whose total stays above 3/4 of its
    8 nv hops at k_O / k_H = 1/13.2, so that the variate named here makes such a ratio."""
    n_tau, kT = 64.0, 8.617333262e-5 * 900.0
    total = 0.75 * 8 * nv * np.exp(-0.2 / kT)  # a lower bound, in units of 1/k32max
    assert 2 ** 6 <= n_tau / 8 * np.exp(0.2 / kT) < 2 ** 7
    assert variate(orc, seed, window, event) / total < 2.0 ** (6 - 29)
    b = fk.Batch([(8, 8, 8, 4.01)], [(nv, 0)], seed, nfrag=(1, 1, 1), precision=1, tracer=True, cap_v=64,
                 n_tau=n_tau, schedule=sched, small_pass=small, lane_form=lane)
    b.set_barriers(0.6, 0.4, 900.0)
    ref = orc.Lattice((8, 8, 8), (1, 1, 1), nv, 0, seed=seed, tracer=True)
    ref.set_rates(0.6, 0.4, 900.0, a_ang=4.01, cap_v=64, n_tau=n_tau, precision=1)
    assert b.info().kernel == (1 if sched == 2 else 0)
    check(b, ref, (window,))
    before = ref.counters()["hops"]
    check(b, ref, (1,))
    assert ref.counters()["hops"] - before > event  # the event happened
    check(b, ref, (3,))


@pytest.mark.parametrize("sched", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
def test_rates_that_underflow_to_zero(fk, orc, prec, sched):
    """O hops at 30 K and 2 eV have the rate 0 in FP64: such an event is never taken,
    also where rounding puts its prefix above those before it."""
    cells, nf, nv, nh = (10, 12, 9), (2, 4, 2), 40, 1500
    b = fk.Batch([(*cells, 4.01)], [(nv, nh)], 4, nfrag=nf, precision=prec, tracer=True, cap_v=64, schedule=sched)
    b.set_barriers(2.0, 0.2, 30.0)
    assert b.info().k64[0] == 0.0 < b.info().k64[3]
    ref = orc.Lattice(cells, nf, nv, nh, seed=4, tracer=True)
    ref.set_rates(2.0, 0.2, 30.0, a_ang=4.01, cap_v=64, precision=prec)
    check(b, ref, (60, 60))


# 4.5 to 20 vacancies per fragment of 12^3 (and 10 x 11 x 13) cells: lists of sixteen fill
# past eight, overflow and refill; one CTA and two slabs
@pytest.mark.parametrize("ctas", [0, 2])
@pytest.mark.parametrize("cells,nf,nv", [((24, 24, 24), (2, 2, 2), 36), ((24, 24, 24), (2, 2, 2), 70),
                                         ((20, 22, 26), (2, 2, 2), 120), ((24, 24, 24), (2, 2, 2), 160)])
def test_lists_of_sixteen(fk, orc, cells, nf, nv, ctas):
    b = fk.Batch([(*cells, 4.01)], [(nv, 2500)], 6, nfrag=nf, precision=1, tracer=True, cap_v=64, cluster_ctas=ctas)
    b.set_barriers(0.6, 0.4, 900.0, field_z=2e7)
    ref = orc.Lattice(cells, nf, nv, 2500, seed=6, tracer=True)
    ref.set_rates(0.6, 0.4, 900.0, Ez=2e7, a_ang=4.01, cap_v=64, precision=1)
    assert b.info().kernel == (2 if ctas else 1)
    check(b, ref, (30, 1, 30, 1))


def test_multigrid_with_planes_that_do_not_divide_by_four(fk, orc):
    """102^3 nodes: the kernels of four planes per thread (2^20 nodes and more), two planes
    and two rows in their last blocks; the next level, 51^3, is the coarsest.  The
    tolerance is that of the smaller lattices."""
    cells = (102, 102, 102)
    b = fk.Batch([(*cells, 4.01)], [(2000, 0)], 3, edge=6, precision=0)
    b.set_barriers(0.7, 0.7, 600.0)
    b.set_electrostatics(eps_r=150.0, q_vac=2.0, refresh_windows=0, cycles=14)
    phi, res = b.solve_potential()
    exact = ps.solve(ps.node_charge(cells, b.records(0)[:, 1], q=2.0), 4.01, 150.0).ravel()
    assert res < 1e-9
    assert np.abs(phi - exact).max() < 1e-8 * np.abs(exact).max()


@pytest.mark.parametrize("sched", [0, 1])
def test_tables_that_grow_within_a_call(fk, orc, sched):
    """A potential written as zeros and solved again after four windows: the refresh
    inside the call needs larger Boltzmann tables and a new plan, and the windows after
    it run with both."""
    cells, nf = (16, 16, 16), (4, 4, 4)
    b = fk.Batch([(*cells, 4.01)], [(90, 200)], 7, nfrag=nf, precision=0, tracer=True, cap_v=64, schedule=sched)
    b.set_barriers(0.6, 0.4, 900.0)
    b.set_electrostatics(eps_r=30.0, refresh_windows=4, cycles=12)
    _, g = b.potential_energy()
    zeros = np.zeros(3 * 16 ** 3, np.int32)
    ref = orc.Lattice(cells, nf, 90, 200, seed=7, tracer=True)
    ref.set_rates(0.6, 0.4, 900.0, a_ang=4.01, cap_v=64)
    done = 0
    for _ in range(3):
        b.write_potential_energy(zeros, g)
        b.run(8)
        u, _ = b.potential_energy()
        assert np.abs(u).max() > 1000
        ref.set_elec(zeros, g)
        ref.run(4)
        ref.set_elec(u, g)
        ref.run(4)
        done += 8
        assert np.array_equal(b.state(), ref.occupancy()) and np.array_equal(b.records(), ref.records())
        assert np.array_equal(b.tracer_field(), ref.tracer_field())
        assert (b.info().hops, b.info().window) == (ref.counters()["hops"], done)
    assert ref.counters()["hops"] > 50
