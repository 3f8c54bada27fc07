"""GPU: direct-sum gravity at the sizes where the tilings change: tile edges,
remainders, aggregates that span several tiles, every tile size of the FP64
path, and piles of different tile sizes in one world."""
import numpy as np
import pytest

from paper_2311_11322_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EPS = 0.3


@pytest.fixture(scope="module")
def dem():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2311_11322_gb300 import dem as D
    return D


def pile(n, precision, seed=0, equal=False):
    """n spheres at random in a cube, no contacts intended: a rod of up to 100 spheres first (it spans tiles), then
    aggregates of 1 to 4 spheres; radii differ unless `equal`."""
    rng = np.random.default_rng(seed + n)
    counts = [min(100, n)]
    while sum(counts) < n:
        counts.append(min(int(rng.integers(1, 5)), n - sum(counts)))
    counts = np.array(counts, np.int32)
    of = np.repeat(np.arange(len(counts)), counts)
    slot = np.arange(n) - np.repeat(np.cumsum(counts) - counts, counts)
    box = 20.0 * n ** (1.0 / 3.0)
    pos = rng.uniform(-box, box, (len(counts), 3))[of]
    pos[:, 0] += 0.5 * slot
    radius = np.full(n, 0.25) if equal else 0.2 + 0.1 * rng.random(len(counts))[of]
    ic = W.PileIC(counts=counts, pos=pos, radius=radius, density=np.full(n, 2500.0))
    return ic, W.Params(G=1e-3, dt=1e-6, kn=1.0, eps=EPS, precision=precision)


def reference(ic, p, pos, sample):
    """Gravity on the sampled spheres and the sum of its terms' magnitudes, in FP64."""
    m = W.sphere_mass(ic.radius, ic.density)
    agg = np.repeat(np.arange(ic.n_agg), ic.counts)
    F, mag = np.zeros((len(sample), 3)), np.zeros(len(sample))
    for k, i in enumerate(sample):
        d = pos - pos[i]
        w = np.where(agg == agg[i], 0.0, m / ((d * d).sum(1) + EPS ** 2) ** 1.5)
        t = p.G * m[i] * w[:, None] * d
        F[k], mag[k] = t.sum(0), np.linalg.norm(t, axis=1).sum()
    return F, mag


def sampled(n):
    return np.unique(np.concatenate([np.arange(min(n, 120)), np.linspace(0, n - 1, 150).astype(int),
                                     np.arange(max(0, n - 70), n)]))


# FP64 tiles: 32 spheres, then 64, 128, 256, 512 as ceil(n / tile) reaches 70
@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 101, 1000, 4416, 4417, 8833, 17665, 35400])
def test_fp64_gravity_tile_sizes(dem, n):
    ic, p = pile(n, W.PRECISION_FP64)
    with dem.World() as w:
        pid = w.add_pile(ic, p)
        w.step(1)
        got, pos = w.read(pid, "SPHERE_FG"), w.read(pid, "SPHERE_POS")
    s = sampled(n)
    F, mag = reference(ic, p, pos, s)
    # a term carries about 10 roundings, a sum of n terms n more, on either side; positions read back are
    # rounded once more than the frame-relative ones summed (1e-16 of the box over the smallest distances)
    err = np.linalg.norm(got[s] - F, axis=1)
    assert np.all(err <= 2 * (n + 20) * 2.0 ** -53 * mag + 1e-12 * mag), float((err / np.maximum(mag, 1e-300)).max())


def test_fp64_tiles_alone_and_in_a_batch_bitwise(dem):
    """Piles of every FP64 tile size in one world give the bits they give alone."""
    piles = [pile(n, W.PRECISION_FP64, seed=7) for n in (40, 900, 4500, 9000, 18000, 36000)]
    alone = []
    for ic, p in piles:
        with dem.World() as w:
            pid = w.add_pile(ic, p)
            w.step(2)
            alone.append(w.read(pid, "SPHERE_FG"))
    with dem.World() as w:
        ids = [w.add_pile(ic, p) for ic, p in piles]
        w.step(2)
        for pid, ref in zip(ids, alone):
            assert np.array_equal(w.read(pid, "SPHERE_FG"), ref)


def test_fp64_budget_keeps_the_large_tiles(dem):
    """A world with a memory budget of the pile's stated footprint still takes the pile and steps it."""
    ic, p = pile(1000, W.PRECISION_FP64)
    need = dem.dem_footprint_bytes(ic.n_sph, ic.n_agg, p.max_contacts, W.PRECISION_FP64)
    with dem.World(budget=need) as w:
        pid = w.add_pile(ic, p)
        w.step(1)
        got, pos = w.read(pid, "SPHERE_FG"), w.read(pid, "SPHERE_POS")
        assert w.bytes() <= need
    s = sampled(1000)
    F, mag = reference(ic, p, pos, s)
    assert np.all(np.linalg.norm(got[s] - F, axis=1) <= 1.5e-12 * mag)


@pytest.mark.parametrize("planet", [0.0, 5.972e24])
@pytest.mark.parametrize("prec", [W.PRECISION_FP64, W.PRECISION_MIXED])
@pytest.mark.parametrize("n", [1, 40, 1000, 4416, 8192, 8193, 12345, 20000])
def test_stated_footprint_covers_a_world_without_a_budget(dem, n, prec, planet):
    """A pile's stated footprint holds for the tiles that a world uses which has no memory budget."""
    ic, p = pile(n, prec)
    p = p.replace(ext_mass=planet, ext_pos=(3.0e7, 0.0, 0.0))
    with dem.World() as w:
        w.add_pile(ic, p)
        w.step(1)
        w.sync()
        assert w.bytes() <= dem.dem_footprint_bytes(ic.n_sph, ic.n_agg, p.max_contacts, prec)


# mixed path: 64-sphere tiles to 8,192 spheres, 256 above; equal masses take their own ring
@pytest.mark.parametrize("equal", [False, True])
@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 129, 1000, 8192, 8193, 12345])
def test_mixed_gravity_tile_edges(dem, n, equal):
    ic, p = pile(n, W.PRECISION_MIXED, seed=3, equal=equal)
    with dem.World() as w:
        pid = w.add_pile(ic, p)
        w.step(2)
        got, pos = w.read(pid, "SPHERE_FG"), w.read(pid, "SPHERE_POS")
    s = sampled(n)
    F, mag = reference(ic, p, pos, s)
    # the mixed path's tolerance, relative to the sum of the terms' magnitudes
    err = np.linalg.norm(got[s] - F, axis=1)
    assert np.all(err <= 1e-5 * mag), float((err / np.maximum(mag, 1e-300)).max())


@pytest.mark.parametrize("tile", [64, 128, 256, 512])
def test_mixed_gravity_tuned_tiles(dem, tile):
    """Every tile size is honoured above 8,192 spheres too."""
    ic, p = pile(9001, W.PRECISION_MIXED, seed=5)
    with dem.World() as w:
        pid = w.add_pile(ic, p)
        w.set_tuning("grav_tile", tile)
        w.step(1)
        got, pos = w.read(pid, "SPHERE_FG"), w.read(pid, "SPHERE_POS")
        assert w.get_tuning("grav_tile") == tile
    s = sampled(9001)
    F, mag = reference(ic, p, pos, s)
    assert np.all(np.linalg.norm(got[s] - F, axis=1) <= 1e-5 * mag)


def test_mixed_large_pile_alone_and_in_a_batch_bitwise(dem):
    """A pile of more than 8,192 spheres gives the same bits whatever else the world holds."""
    piles = [pile(n, W.PRECISION_MIXED, seed=9, equal=n == 700) for n in (9000, 700, 15000)]
    with dem.World() as w:
        pid = w.add_pile(*piles[0])
        w.step(3)
        alone = w.read(pid, "SPHERE_FG"), w.read(pid, "VEL")
    with dem.World() as w:
        ids = [w.add_pile(ic, p) for ic, p in piles]
        w.step(3)
        assert np.array_equal(w.read(ids[0], "SPHERE_FG"), alone[0])
        assert np.array_equal(w.read(ids[0], "VEL"), alone[1])


@pytest.mark.parametrize("precision", [W.PRECISION_MIXED, W.PRECISION_FP64])
@pytest.mark.parametrize("n_agg", [1, 31, 128, 129, 512, 513, 1700])
def test_pile_reductions_over_blocks_and_chunks(dem, n_agg, precision):
    """COM frame, mean velocity and the planet's reaction of piles of one block, one chunk and several: after a step
    the frame is the drifted COM and the planet's acceleration the sum of its forces."""
    rng = np.random.default_rng(n_agg)
    pos = rng.uniform(-50, 50, (n_agg, 3))
    ic = W.PileIC(counts=np.ones(n_agg, np.int32), pos=pos, radius=0.1 + 0.1 * rng.random(n_agg),
                  density=np.full(n_agg, 2500.0), vel=rng.standard_normal((n_agg, 3)))
    p = W.Params(G=1e-6, dt=1e-3, kn=1.0, eps=0.5, precision=precision, ext_mass=1e9, ext_pos=(3e3, 1e3, -2e3),
                 ext_vel=(5.0, -7.0, 11.0))
    with dem.World() as w:
        pid = w.add_pile(ic, p)
        w.step(1)
        com, fe = w.read(pid, "COM"), w.read(pid, "FORCE_EXT")
        planet, frame, M = w.read(pid, "PLANET"), w.read(pid, "FRAME"), w.read(pid, "MASS")
        assert w.info(pid)["steps"] == 1
    # mixed sums are float-float with FP32 masses: 2^-24 of the largest term
    tol = 1e-13 if precision == W.PRECISION_FP64 else 2.0 ** -23
    assert np.allclose(frame[:3], (M[:, None] * com).sum(0) / M.sum(), rtol=0, atol=50 * tol)
    assert np.allclose(frame[3:], (M[:, None] * ic.vel).sum(0) / M.sum(), rtol=0, atol=5 * tol)
    # n terms of a sum in float-float (2^-44) or FP64
    react = -fe.sum(0) / p.ext_mass
    assert np.allclose(planet[6:], react, rtol=0, atol=1e-11 * np.abs(fe).sum() / p.ext_mass)
    m = W.sphere_mass(ic.radius, ic.density)
    P = np.array(p.ext_pos) + p.dt * np.array(p.ext_vel)
    d = P - com
    ref = (p.G * p.ext_mass * m / (d * d).sum(1) ** 1.5)[:, None] * d
    assert np.all(np.linalg.norm(fe - ref, axis=1) <= 1e-13 * np.linalg.norm(ref, axis=1) + 1e-300)


# tree depths 2 .. 5: leaf counts below, at and above one scan block; groups with a remainder
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("n", [1, 2, 33, 300, 1025, 2049, 8300, 17001])
def test_tree_gravity_small_angle_is_the_direct_sum(dem, n, order):
    """With a small opening angle the accepted cells' expansions are exact to far below the mixed tolerance (their
    relative error is about theta^(order + 1)), so the tree, its leaves and its moments must give the direct sum."""
    ic, p = pile(n, W.PRECISION_MIXED, seed=11)
    with dem.World() as w:
        w.set_tuning("grav_theta", 0.05 if order == 4 else 0.01)
        w.set_tuning("grav_order", order)
        pid = w.add_pile(ic, p)
        w.step(1)
        got, pos = w.read(pid, "SPHERE_FG"), w.read(pid, "SPHERE_POS")
    s = sampled(n)
    F, mag = reference(ic, p, pos, s)
    err = np.linalg.norm(got[s] - F, axis=1)
    assert np.all(err <= 1e-5 * mag), float((err / np.maximum(mag, 1e-300)).max())


# tree depths 2 (53 and 81 spheres), 3 and 4
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("k", [3, 7, 40, 300, 1200])
def test_tree_expansions_of_accepted_cells(dem, k, order):
    """Moments and expansions by themselves: seven rods of k spheres in corners of a cube, pointing at the eighth
    corner, where one aggregate of 32 spheres (no forces of its own) probes them.  Its group is the first of the leaf
    order, and at this angle it accepts each rod whole, as the one cell of the walk's first level that holds it."""
    rng = np.random.default_rng(k)
    edge, b, eps = 100.0, 6.0, 0.01

    def ball(m, radius):
        v = rng.standard_normal((m, 3))
        return v * (radius * rng.random(m) ** (1 / 3) / np.linalg.norm(v, axis=1))[:, None]
    pos, rod = [ball(32, 3.0)], [np.full(32, -1)]
    for c in range(1, 8):
        corner = edge * np.array([c & 1, c >> 1 & 1, c >> 2 & 1], float)
        end = np.where(np.arange(k) % 3 == 0, -0.9, 0.9)      # a third at one end: all ranks of moments
        pos.append(corner + b * end[:, None] * corner / np.linalg.norm(corner) + ball(k, 0.08 * b))
        rod.append(np.full(k, c))
    pos, rod = np.concatenate(pos), np.concatenate(rod)
    n = len(pos)
    ic = W.PileIC(counts=np.concatenate([[32], np.ones(7 * k, int)]).astype(np.int32), pos=pos,
                  radius=rng.uniform(0.001, 0.0015, n), density=np.full(n, 2500.0))
    p = W.Params(G=1.0, dt=1e-9, kn=1.0, eps=eps, precision=W.PRECISION_MIXED)
    with dem.World() as w:
        w.set_tuning("grav_theta", 0.45)
        w.set_tuning("grav_order", order)
        pid = w.add_pile(ic, p)
        w.step(1)
        got, x = w.read(pid, "SPHERE_FG")[:32], w.read(pid, "SPHERE_POS")
    m = W.sphere_mass(ic.radius, ic.density)
    F, mag, tol = np.zeros((32, 3)), np.zeros(32), np.zeros(32)
    for c in range(1, 8):
        mine = rod == c
        com = (m[mine, None] * x[mine]).sum(0) / m[mine].sum()
        radius = np.linalg.norm(x[mine] - com, axis=1).max()
        d = x[mine][None] - x[:32, None]
        r = np.linalg.norm(d, axis=2)
        F += m[:32, None] * ((m[mine] / (r * r + eps ** 2) ** 1.5)[:, :, None] * d).sum(1)
        part = m[:32] * (m[mine] / (r * r)).sum(1)
        q = radius / np.linalg.norm(com - x[:32], axis=1)
        # the ranks left out: (n + 1) q^n of M / d^2 each, M / d^2 at most (1 + q)^2 of the terms' sum
        tol += part * (1 + q) ** 2 * sum((j + 1) * q ** j for j in range(order + 1, 40))
        mag += part
    err = np.linalg.norm(got - F, axis=1)
    # FP32: some ten roundings of 2^-24 on the way to each term, the sums, and the positions
    assert np.all(err <= tol + 3e-6 * mag), float((err / mag).max())
    if order == 2:
        assert np.all(err > 1e-5 * mag)      # the rods were not summed sphere by sphere


def test_tree_piles_of_different_depths_alone_and_in_a_batch_bitwise(dem):
    piles = [pile(n, W.PRECISION_MIXED, seed=13) for n in (3, 270, 2100, 9000, 40)]

    def run(sel):
        with dem.World() as w:
            w.set_tuning("grav_theta", 0.6)
            ids = [w.add_pile(*piles[k]) for k in sel]
            w.step(2)
            return [w.read(pid, "SPHERE_FG") for pid in ids]
    alone = [run([k])[0] for k in range(len(piles))]
    for got, ref in zip(run(range(len(piles))), alone):
        assert np.array_equal(got, ref)


@pytest.mark.parametrize("eps", [0.0, 0.5])
@pytest.mark.parametrize("ids", ["contiguous", "shuffled"])
@pytest.mark.parametrize("n", [2, 127, 129, 512, 513, 1025, 5003])
def test_noalloc_gravity_parts_and_masks(dem, n, ids, eps):
    """The caller-owned gravity call at the edges of its blocks, tiles and parts, with aggregate ids in order and in
    none, softened and not (two spheres of different aggregates coincide: no force between them)."""
    import torch
    rng = np.random.default_rng(n)
    pos = rng.uniform(-200.0, 200.0, (n, 3)).astype(np.float32)
    agg = (np.arange(n) // 3).astype(np.int32)
    if ids == "shuffled":
        agg = rng.permutation(agg) - 5
    if n > 6:
        pos[-1] = pos[0]
        agg[-1], agg[0] = 1000000, -1000000
    m = W.sphere_mass(rng.uniform(1.0, 3.0, n), 2500.0)
    pm = torch.from_numpy(np.concatenate([pos, m.astype(np.float32)[:, None]], 1)).cuda()
    tm, ta = torch.from_numpy(m).cuda(), torch.from_numpy(agg).cuda()
    out = torch.full((n, 4), float("nan"), dtype=torch.float64, device="cuda")
    import ctypes as C
    rc = dem.load().dem_gravity_noalloc(pm.data_ptr(), C.c_void_p(tm.data_ptr()), ta.data_ptr(), n, 1.0, eps,
                                        C.c_void_p(out.data_ptr()), torch.cuda.current_stream().cuda_stream, None, 0)
    assert rc == dem.DEM_OK
    got = out.cpu().numpy()[:, :3]
    for i in sampled(n):
        d = pos.astype(float) - pos[i].astype(float)
        r2 = (d * d).sum(1) + eps ** 2
        w = np.where((agg == agg[i]) | (r2 == 0), 0.0, m / np.where(r2 == 0, 1.0, r2) ** 1.5)
        t = m[i] * w[:, None] * d
        assert np.linalg.norm(got[i] - t.sum(0)) <= 1e-5 * np.linalg.norm(t, axis=1).sum()


def test_planet_pile_comes_and_goes(dem):
    """A planet pile added to and removed from a world without planets: every pile steps as it does alone, and later
    piles are not charged for a planet's forces."""
    sets = []
    for n, mass in ((900, 0.0), (700, 5.972e24), (333, 0.0)):
        ic, p = pile(n, W.PRECISION_MIXED, seed=n)
        sets.append((ic, p.replace(ext_mass=mass, ext_pos=(3.0e7, 1.0e6, 0.0), ext_vel=(0.0, 9.0e3, 0.0))))
    fields = ("COM", "VEL", "QUAT", "FORCE_EXT", "TORQUE", "SPHERE_FG")
    alone = []
    for (ic, p), steps in zip(sets, (9, 3, 6)):
        with dem.World() as w:
            pid = w.add_pile(ic, p)
            w.step(steps)
            alone.append({f: w.read(pid, f) for f in fields})
    with dem.World() as w:
        a = w.add_pile(*sets[0])
        w.step(3)
        b = w.add_pile(*sets[1])       # the world's first planet
        w.step(3)
        assert all(np.array_equal(w.read(b, f), alone[1][f]) for f in fields)
        assert np.abs(alone[1]["FORCE_EXT"]).max() > 0
        w.remove(b)
        c = w.add_pile(*sets[2])
        w.step(3)
        b = w.add_pile(*sets[1])       # and again, beside both
        w.step(3, piles=[b, c])
        for pid, ref in ((a, alone[0]), (b, alone[1]), (c, alone[2])):
            assert all(np.array_equal(w.read(pid, f), ref[f]) for f in fields)
    big = pile(30_000, W.PRECISION_MIXED)
    held = []
    for planet_first in (False, True):
        with dem.World() as w:
            pid = w.add_pile(*sets[1 if planet_first else 0])
            w.step(1)
            w.remove(pid)
            w.add_pile(*big)
            w.step(1)
            held.append(w.bytes())
    assert held[1] < held[0] + 32 * 900 + 4096    # the first pile's own spheres at most
