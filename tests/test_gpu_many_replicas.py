"""Which kernel a batch of several replicas runs in: clusters as large as the GPU can
place all of them at once, one CTA each where not all of a batch's dense replicas
can have a cluster, the colour-phase passes where the resident kernels would take
several waves or draw for mostly empty fragments; and the same trajectories on
each side of the lines."""
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


def batch(fk, n, cells, nf, nv, nh, prec, **kw):
    b = fk.Batch([(*cells, 4.01)] * n, [(nv, nh)] * n, 21, nfrag=nf, precision=prec, cap_v=32, **kw)
    b.set_barriers(0.6, 0.4, 900.0)
    return b, [(b.info(r).kernel, b.info(r).ctas) for r in range(n)]


def same(orc, b, cells, nf, nv, nh, prec, windows, replicas):
    for w in windows:
        b.run(w)
    for r in replicas:
        ref = orc.Lattice(cells, nf, nv, nh, seed=21, replica=r)
        ref.set_rates(0.6, 0.4, 900.0, a_ang=4.01, cap_v=32, precision=prec)
        ref.run(sum(windows))
        assert np.array_equal(b.state(r), ref.occupancy()) and np.array_equal(b.records(r), ref.records()), r
        assert b.info(r).hops == ref.counters()["hops"] > 0


@pytest.mark.parametrize("prec", [0, 1])
def test_clusters_shrink_until_all_run_at_once(fk, orc, prec):
    cells, nf, nv, nh = (64, 64, 64), (16, 16, 16), 786, 8000
    ctas = []
    for n in (1, 12, 40):
        b, kind = batch(fk, n, cells, nf, nv, nh, prec)
        assert set(kind) == {(2, kind[0][1])}
        ctas.append(kind[0][1])
        same(orc, b, cells, nf, nv, nh, prec, (6, 1), (0, n - 1))
        b.close()
    # 40 clusters of 4 CTAs would need more SMs than there are, 12 of 16 as well
    assert ctas[0] == 16 > ctas[1] > ctas[2] >= 2


@pytest.mark.parametrize("prec", [0, 1])
def test_dense_replicas_move_to_clusters_together_or_not(fk, orc, prec):
    cells, nf, nv, nh = (32, 32, 32), (8, 8, 8), 983, 2000
    for n, kernel in ((2, 2), (152, 1)):
        b, kind = batch(fk, n, cells, nf, nv, nh, prec)
        assert {k for k, _ in kind} == {kernel}
        same(orc, b, cells, nf, nv, nh, prec, (5, 4), (0, n - 1))
        b.close()


# plain: 1400 x 1728 mostly empty fragments to draw for; mixed: clusters of 128^3 in more than one wave
@pytest.mark.parametrize("prec,n,cells,nf,nv", [(0, 1400, (24, 24, 24), (12, 12, 12), 60),
                                                (1, 32, (128, 128, 128), (32, 32, 32), 6291)])
def test_large_batches_take_the_passes(fk, orc, prec, n, cells, nf, nv):
    b, kind = batch(fk, n, cells, nf, nv, 50 * nv, prec)
    assert set(kind) == {(0, 0)}
    same(orc, b, cells, nf, nv, 50 * nv, prec, (3, 2), (n - 1,))
    b.close()
    b, kind = batch(fk, 4, cells, nf, nv, 50 * nv, prec)
    assert all(k > 0 for k, _ in kind)
    same(orc, b, cells, nf, nv, 50 * nv, prec, (3, 2), (3,))
