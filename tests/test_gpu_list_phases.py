"""GPU: the phases of a candidate-list rebuild.  Results must not depend on
how many blocks take part in a rebuild, on how long they wait for one another,
on what other streams run, nor on how many spheres share a cell."""
import numpy as np
import pytest

from paper_2311_11322_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("COM", "VEL", "QUAT", "OMEGA", "ACC", "TORQUE", "SPHERE_FC", "CONTACTS")


@pytest.fixture(scope="module")
def dem():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2311_11322_gb300 import dem as D
    return D


def piles(prec):
    """A pile that rebuilds often, a larger one with self-gravity that seldom does, one aggregate alone."""
    fast = W.random_cluster(8, n_agg=60, box=5.0, precision=prec)
    out = [fast]
    for n, seed in ((20_011, 9), (5, 2)):
        ic, p = W.dense_lattice(n_spheres=n, seed=seed, precision=prec)
        out.append((ic, p.replace(max_contacts=fast[1].max_contacts, G=6.67430e-11)))
    return out


def state(w, pid):
    return {f: w.read(pid, f) for f in FIELDS}


def same(got, ref):
    for f in FIELDS:
        assert np.array_equal(got[f], ref[f]), f


@pytest.mark.parametrize("skin", [0.02, 0.0])
@pytest.mark.parametrize("prec", [W.PRECISION_FP64, W.PRECISION_MIXED])
def test_waits_that_run_out_change_nothing(dem, prec, skin):
    """A block that gives up its wait leaves the rest of the rebuild to those still working: with waits that end
    after no, one or a few polls every pile, rebuilding or not, takes exactly the steps it takes otherwise."""
    ref = None
    for wait in (None, 0, 1, 40):
        with dem.World() as w:
            w.set_tuning("skin", skin)
            if wait is not None:
                w.set_tuning("list_wait", wait)
                assert w.get_tuning("list_wait") == wait
            ids = [w.add_pile(ic, p) for ic, p in piles(prec)]
            w.step(25)
            w.sync()
            assert all(not w.flags(k) & (1 | 2 | 16) for k in ids)
            got = [state(w, k) for k in ids]
            rebuilds = [w.info(k)["rebuilds"] for k in ids]
        if ref is None:
            ref, rebuilds0 = got, rebuilds
            assert skin == 0.0 or rebuilds[1] < rebuilds[0]   # some steps rebuild one pile and not the other
        for g, r in zip(got, ref):
            same(g, r)
        assert rebuilds == rebuilds0


def test_list_wait_is_checked(dem):
    with dem.World() as w:
        for bad in (-1, 2.0 ** 31):
            with pytest.raises(dem.DemError):
                w.set_tuning("list_wait", bad)


@pytest.mark.parametrize("prec", [W.PRECISION_FP64, W.PRECISION_MIXED])
def test_worlds_that_share_the_gpu(dem, prec):
    """Worlds on streams of their own, each rebuilding its lists in every step, give what they give alone."""
    sets = [W.dense_lattice(n_spheres=n, seed=n, precision=prec, speed=0.01) for n in (30_000, 150_000, 1_001)]
    alone = []
    for ic, p in sets:
        with dem.World() as w:
            w.set_tuning("skin", 0.0)
            pid = w.add_pile(ic, p)
            w.step(30)
            alone.append(state(w, pid))
    worlds = [dem.World() for _ in sets]
    try:
        ids = []
        for w, (ic, p) in zip(worlds, sets):
            w.set_tuning("skin", 0.0)
            ids.append(w.add_pile(ic, p))
        for _ in range(6):
            for w in worlds:
                w.step(5)
        for w, pid, ref in zip(worlds, ids, alone):
            same(state(w, pid), ref)
            assert w.info(pid)["rebuilds"] == 30
    finally:
        for w in worlds:
            w.close()
