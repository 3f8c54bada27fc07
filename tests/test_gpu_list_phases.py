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


@pytest.mark.parametrize("prec", [W.PRECISION_FP64, W.PRECISION_MIXED])
@pytest.mark.parametrize("n", [28, 3_001, 40_000])
def test_cells_of_any_population(dem, prec, n):
    """Cells far larger than the spheres (the whole pile in a few of them) give the bits of ordinary cells."""
    ic, p = W.dense_lattice(n_spheres=n, seed=n, precision=prec, speed=0.01)
    got = []
    for cell in (0.0, 1.0e4):
        with dem.World() as w:
            w.set_tuning("skin", 0.02)
            pid = w.add_pile(ic, p.replace(cell_size=cell))
            w.step(20)
            w.sync()
            info = w.info(pid)
            assert info["rebuilds"] > 1 and not int(info["flags"]) & (1 | 2 | 16)
            got.append(state(w, pid))
            if cell:
                assert info["nx"] * info["ny"] * info["nz"] == 27
    same(got[1], got[0])


@pytest.mark.parametrize("prec", [W.PRECISION_FP64, W.PRECISION_MIXED])
def test_a_boulder_among_grains(dem, prec):
    """One sphere 60 times as large as the 40,000 others makes cells that hold thousands of them: the pile steps
    without a flag, and the first step's contacts are those of a search over all pairs."""
    spatial = pytest.importorskip("scipy.spatial")
    ic, p = W.dense_lattice(n_spheres=40_000, seed=3, precision=prec)
    R = 60.0
    top = ic.pos[:, 2].max() + 1.0 + R + 3.0       # clear of the grains
    ic.counts = np.append(ic.counts, 1).astype(np.int32)
    ic.pos = np.vstack([ic.pos, [[0.0, 0.0, top]]])
    ic.radius = np.append(ic.radius, R)
    ic.density = np.append(ic.density, 2500.0)
    ic.vel = np.vstack([ic.vel, np.zeros((1, 3))])
    ic.omega = np.vstack([ic.omega, np.zeros((1, 3))])
    with dem.World() as w:
        w.set_tuning("skin", 0.002)    # (0.1 of the boulder's radius would list hundreds of neighbours per grain)
        pid = w.add_pile(ic, p)
        info = w.info(pid)
        assert info["cell"] > 2 * R
        w.step(1)
        w.sync()
        pairs, _ = w.contacts(pid)
        pos = w.read(pid, "SPHERE_POS")
        assert not w.flags(pid) & (1 | 2 | 16)
        w.step(3)
        w.sync()
        assert not w.flags(pid) & (1 | 2 | 16)
    agg = np.repeat(np.arange(len(ic.counts)), ic.counts)
    near = spatial.cKDTree(pos[:-1]).query_pairs(2.0, output_type="ndarray")
    near = near[agg[near[:, 0]] != agg[near[:, 1]]]
    gap = 2.0 - np.linalg.norm(pos[near[:, 0]] - pos[near[:, 1]], axis=1)
    # pairs that only just touch (within the rounding of the positions) may be on either side
    sure = {tuple(sorted(map(int, q))) for q, g in zip(near, gap) if g > 1e-6}
    maybe = {tuple(sorted(map(int, q))) for q in near}
    got = set(pairs)
    assert len(sure) > 40_000 and sure <= got <= maybe
