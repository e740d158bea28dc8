"""Calls that meet an allocator without room: a batch either goes on without the
memory (the colour-phase passes need none of their own) or refuses to run until
its rates are set again; nothing is launched on a buffer that is not there."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CELLS, NV, NH = (12, 12, 12), 20, 40
VV = [(2, 0.343), (4, 0.235), (6, 0.200)]


@pytest.fixture(scope="module")
def fk():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2004_09081_gb300 import fkmc
    fkmc.load()
    return fkmc


class Limited:
    """Torch memory through the ABI's callback: records the sizes asked for, and
    from `limit` on gives nothing after `fail_from` requests."""

    def __init__(self, fk):
        self.inner = fk.TorchAllocator()
        self.sizes, self.fail_from = [], None
        self.c_alloc = fk.kmc_alloc_fn(self._alloc)
        self.c_free = self.inner.c_free

    def limit(self, fail_from):
        self.sizes, self.fail_from = [], fail_from

    def _alloc(self, ctx, n):
        self.sizes.append(n)
        if self.fail_from is not None and len(self.sizes) > self.fail_from:
            return None
        return self.inner._alloc(ctx, n)


def lattice(fk, prec, al, **kw):
    b = fk.Batch([(*CELLS, 4.01)], [(NV, NH)], 8, edge=4, precision=prec, cap_v=32, alloc=al, **kw)
    return b


def reference(orc, prec, windows, site=False):
    ref = orc.Lattice(CELLS, None, NV, NH, seed=8, edge=4)
    if site:
        ref.set_site_energy(vv=VV)
    ref.set_rates(0.7, 0.35, 800.0, a_ang=4.01, cap_v=32, precision=prec)
    ref.run(windows)
    return ref


def same(b, ref):
    assert np.array_equal(b.state(), ref.occupancy())
    assert np.array_equal(b.records(), ref.records())
    assert b.info().hops == ref.counters()["hops"] > 0


# the first request (first draws or site map), and each later one
@pytest.mark.parametrize("fail_from", [0, 1, 2])
@pytest.mark.parametrize("prec", [0, 1])
def test_without_the_resident_buffers_the_passes_run(fk, orc, prec, fail_from):
    al = Limited(fk)
    b = lattice(fk, prec, al)
    b.set_grains(4, 1, 0.2)
    b.set_barriers(0.7, 0.35, 800.0)  # grains: no resident replica, no buffers
    al.limit(fail_from)
    b.set_grains(0)
    need = 3 - prec  # draws (plain form), site map, records
    assert b.info().kernel == (0 if fail_from < need else 1)
    b.run(15)
    al.limit(None)
    same(b, reference(orc, prec, 15))
    b.set_barriers(0.7, 0.35, 800.0)
    assert b.info().kernel == 1
    b.run(10)
    same(b, reference(orc, prec, 25))


@pytest.mark.parametrize("fail_from", [0, 1])
def test_resident_only_batch_is_refused_without_its_buffers(fk, orc, fail_from):
    al = Limited(fk)
    b = lattice(fk, 1, al, schedule=2)
    al.limit(fail_from)
    with pytest.raises(fk.KmcError) as e:
        b.set_barriers(0.7, 0.35, 800.0)
    assert e.value.code == fk.FKMC_ENOMEM
    with pytest.raises(fk.KmcError) as e:
        b.run(1)
    assert e.value.code == fk.FKMC_ESTATE
    al.limit(None)
    b.set_barriers(0.7, 0.35, 800.0)
    b.run(15)
    same(b, reference(orc, 1, 15))


def test_failed_energy_tables_stop_the_batch(fk, orc):
    """kmc_set_site_energy with an allocator that fails from each request on: where
    the call fails before the interactions are on, the batch runs on without them;
    where the Boltzmann tables fail, it is refused until the rates are set."""
    seen = set()
    for k in range(8):
        al = Limited(fk)
        b = lattice(fk, 0, al)
        b.set_barriers(0.7, 0.35, 800.0)
        al.limit(k)
        try:
            b.set_site_energy(VV)
            seen.add("set")
        except fk.KmcError as e:
            assert e.code == fk.FKMC_ENOMEM
            try:
                b.run(40)
                seen.add("runs without")
                al.limit(None)
                same(b, reference(orc, 0, 40))
                continue
            except fk.KmcError as e2:
                assert e2.code == fk.FKMC_ESTATE
                seen.add("refused")
        al.limit(None)
        b.set_barriers(0.7, 0.35, 800.0)
        b.run(40)
        same(b, reference(orc, 0, 40, site=True))
    assert seen == {"set", "runs without", "refused"}


def test_read_outs_without_a_device_buffer(fk, orc):
    al = Limited(fk)
    b = lattice(fk, 1, al)
    b.set_barriers(0.7, 0.35, 800.0)
    b.run(15)
    ref = reference(orc, 1, 15)
    al.limit(0)
    same(b, ref)
    assert al.sizes  # the buffer was asked for
    al.limit(None)
    same(b, ref)


def plan(b):
    i = b.info()
    return i.kernel, i.ctas, i.draw_phases, i.draw_events


def test_own_potential_alone_outgrows_the_planned_tables(fk, orc):
    """An all-zero potential written with a larger own-potential table needs larger
    Boltzmann tables, and with them a new plan: the shared memory that was planned
    for the smaller ones does not hold them."""
    cells, nf, nv = (32, 32, 32), (8, 8, 8), 200
    b = fk.Batch([(*cells, 4.01)], [(nv, 0)], 5, nfrag=nf, precision=0, cap_v=32)
    b.set_electrostatics(eps_r=100.0, refresh_windows=0)
    u = np.zeros(3 * 32 ** 3, np.int32)
    g = np.full((3, 8), -100, np.int32)
    b.write_potential_energy(u, g)
    b.set_barriers(0.6, 0.6, 900.0)
    small = plan(b)
    g[0, 0] = -400000  # one direction closed by 20 eV
    b.write_potential_energy(u, g)
    grown = plan(b)
    b.set_barriers(0.6, 0.6, 900.0)
    assert grown == plan(b) != small
    b.write_potential_energy(u, g)
    b.run(60)
    ref = orc.Lattice(cells, nf, nv, 0, seed=5)
    ref.set_elec(u, g)
    ref.set_rates(0.6, 0.6, 900.0, a_ang=4.01, cap_v=32)
    ref.run(60)
    same(b, ref)


def null_reference(orc, steps, cells=CELLS, nv=NV, nh=NH, replica=0):
    ref = orc.Lattice(cells, None, nv, nh, seed=8, edge=4, replica=replica)
    ref.set_rates(0.7, 0.35, 800.0, a_ang=4.01, cap_v=32, precision=1)
    ref.null_run(steps, 8)
    return ref


def test_null_event_form_asks_for_what_its_steps_need(fk, orc):
    """Claims, vacancies and picks, and a word per vacancy and 32 bytes per step where
    one launch makes the steps."""
    al = Limited(fk)
    b = lattice(fk, 1, al)
    b.set_barriers(0.7, 0.35, 800.0)
    al.limit(None)
    b.run_null(3, 8)
    assert sum(al.sizes) < 8 * b.nsite() + 100 * NV + 4096
    al.limit(None)
    b.run_null(50, 8)
    assert sum(al.sizes) < 50 * 32 + 4096
    same(b, null_reference(orc, 53))


def test_null_event_form_beyond_one_launch(fk, orc):
    """More replicas than the GPU holds CTAs for: launches per step, no step log."""
    n, cells, nv, nh = 5000, (4, 4, 4), 3, 20
    al = Limited(fk)
    b = fk.Batch([(*cells, 4.01)] * n, [(nv, nh)] * n, 8, edge=4, precision=1, cap_v=32, alloc=al)
    b.set_barriers(0.7, 0.35, 800.0)
    al.limit(None)
    b.run_null(20, 8)
    assert sum(al.sizes) < n * (8 * b.nsite() + 100 * nv + 100)
    for r in (0, 1, n - 1):
        ref = null_reference(orc, 20, cells, nv, nh, r)
        assert np.array_equal(b.state(r), ref.occupancy()) and np.array_equal(b.records(r), ref.records())


def test_null_event_form_at_every_failing_request(fk, orc):
    done = 0
    for k in range(12):
        al = Limited(fk)
        b = lattice(fk, 1, al)
        b.set_barriers(0.7, 0.35, 800.0)
        al.limit(k)
        try:
            b.run_null(20, 8)
        except fk.KmcError as e:
            assert e.code == fk.FKMC_ENOMEM
            continue
        al.limit(None)
        same(b, null_reference(orc, 20))
        done += 1
    assert done >= 3  # without both buffers of the one launch, without its log, with everything


def test_null_event_form_after_failed_calls(fk, orc):
    """One request more granted by each call: what the earlier ones left is used, and
    nothing that is missing."""
    al = Limited(fk)
    b = lattice(fk, 1, al)
    b.set_barriers(0.7, 0.35, 800.0)
    for k in range(10):
        al.limit(1)
        try:
            b.run_null(20, 8)
        except fk.KmcError as e:
            assert e.code == fk.FKMC_ENOMEM
    al.limit(None)
    assert b.info().null_steps >= 40
    same(b, null_reference(orc, b.info().null_steps))
