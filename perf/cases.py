"""The work a user has this framework do, as a set of measurable cases.

Every case but one advances rubble piles through ``dem.World``: make the pile(s) once, then step and read
the new state back, which is what a simulation driver does.  A pass is a handful of steps followed by that
read (drivers read every few steps, not after each one).  Kinds:

  cloud      bonded aggregates drifting in a ball: the collapse runs (few contacts, direct or tree gravity)
  settled    a dense ellipsoid with nearly every neighbour in contact, gravity and a YORP spin ramp
  encounter  a loose lattice pile passing an Earth-mass point (the tidal-encounter requests)
  batch      many independent piles of lognormal sizes advanced by one call
  request    one pile admitted to a world, stepped, read back and removed again (a served simulation);
             a dense lattice without self-gravity, so contacts and the list build are the work
  field      dem_gravity_noalloc: gravity of one set of spheres in the caller's own buffers

Outputs are the aggregates' new state and acceleration (and the stored torque where contacts carry it).
Piles of the mixed path form forces in FP32, so what follows from one step's forces is handed on as FP32;
positions and orientations, which the library keeps to 48 bits, stay FP64.  Piles of the FP64 path stay FP64.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

G_SI = 6.67430e-11
EARTH_MASS, EARTH_RADIUS = 5.972e24, 6.371e6

_R3, _R2 = math.sqrt(3.0), 1.0 / math.sqrt(2.0)
# member offsets in units of the sphere radius (touching spheres)
SHAPES = {
    "single": [(0, 0, 0)],
    "dumbbell": [(1, 0, 0), (-1, 0, 0)],
    "rod3": [(-2, 0, 0), (0, 0, 0), (2, 0, 0)],
    "tetra": [(_R2, _R2, _R2), (_R2, -_R2, -_R2), (-_R2, _R2, -_R2), (-_R2, -_R2, _R2)],
    "square": [(1, 1, 0), (1, -1, 0), (-1, 1, 0), (-1, -1, 0)],
    "rod4": [(-3, 0, 0), (-1, 0, 0), (1, 0, 0), (3, 0, 0)],
    "diamond": [(0, 1, 0), (0, -1, 0), (_R3, 0, 0), (-_R3, 0, 0)],
    "cube8": [(i, j, k) for i in (-1, 1) for j in (-1, 1) for k in (-1, 1)],
}
MIXES = {
    "simple": ("dumbbell", "rod3", "tetra", "square"),              # the collapse benchmark
    "grains": ("dumbbell", "diamond", "rod4", "tetra", "cube8"),    # the paper's profiling runs
    "tetra": ("tetra",),                                            # batches, encounters
}


# ---------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one small pile (250 grains), the size of a quick experiment: launches and latency are all there is
        dict(name="cloud-1k", kind="cloud", n=1000, mix="tetra", s=1.0, sigma=0.06, spacing=1.5, precision="mixed", theta=0.0,
             steps=20),
        # the same experiment in all-FP64, the default of the small configuration
        dict(name="cloud-1k-fp64", kind="cloud", n=1000, mix="tetra", s=1.0, sigma=0.06, spacing=1.5, precision="fp64",
             theta=0.0, steps=20),
        # a tidal encounter at the median size of the served trace
        dict(name="encounter-7k", kind="encounter", n=7466, s=1.0, sigma=0.06, precision="mixed", theta=0.0, steps=20),
        # the paper's 2e4-sphere profiling collapse: equal 50 m spheres in five grain shapes
        dict(name="cloud-20k", kind="cloud", n=20_000, mix="grains", s=50.0, sigma=0.0, spacing=1.5, precision="mixed",
             theta=0.0, steps=20),
        # a mid-size collapse in all-FP64 (reference runs), at an odd count
        dict(name="cloud-12k-fp64", kind="cloud", n=12_345, mix="simple", s=5.0, sigma=0.2, spacing=2.5, precision="fp64",
             theta=0.0, steps=5),
        # the benchmark: collapse of 100,000 spheres by direct sum
        dict(name="cloud-100k", kind="cloud", n=100_000, mix="simple", s=5.0, sigma=0.2, spacing=2.5, precision="mixed",
             theta=0.0, steps=10),
        # the same collapse at an odd count with tree gravity, the paper's method
        dict(name="cloud-100k-tree", kind="cloud", n=99_991, mix="simple", s=5.0, sigma=0.2, spacing=2.5, precision="mixed",
             theta=0.7, steps=20),
        # a spun-up settled pile: dense contacts, direct sum, the largest single pile
        dict(name="settled-200k", kind="settled", n=200_000, s=1.0, precision="mixed", theta=0.0, steps=4),
        # a settled pile of odd size under tree gravity, the cheap way to run such a pile for long
        dict(name="settled-50k-tree", kind="settled", n=50_003, s=1.0, precision="mixed", theta=0.5, steps=20),
        # a parameter study: 256 piles of 500 to 20,000 spheres advanced together
        dict(name="batch-256", kind="batch", piles=256, median=3000, s=1.0, sigma=0.06, precision="mixed", steps=10),
        # a served contact-dominated simulation of a million spheres: admit, step, read, remove
        dict(name="request-1m", kind="request", n=1_048_576, s=1.0, precision="mixed", steps=100),
        # a host program's own gravity call on its own buffers
        dict(name="field-20k", kind="field", n=20_001, s=5.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cloud", "cloud", "fp64", "tree", "settled", "encounter", "batch", "request", "field"])
    if kind == "cloud":
        n = _log(rng, 500, 100_000)
        mix, s, sigma, spacing = rng.choice([("simple", 5.0, 0.2, 2.5), ("grains", 50.0, 0.0, 1.5), ("tetra", 1.0, 0.06, 1.5)])
        return dict(kind="cloud", n=n, mix=mix, s=s, sigma=sigma, spacing=spacing, precision="mixed", theta=0.0, steps=10)
    if kind == "fp64":
        return dict(kind="cloud", n=_log(rng, 500, 20_000), mix=rng.choice(["simple", "tetra"]), s=1.0, sigma=0.1,
                    spacing=rng.choice([1.5, 2.5]), precision="fp64", theta=0.0, steps=5)
    if kind == "tree":
        return dict(kind=rng.choice(["cloud", "settled"]), n=_log(rng, 4000, 200_000), mix="simple", s=5.0, sigma=0.2,
                    spacing=2.5, precision="mixed", theta=rng.choice([0.5, 0.6, 0.7]), steps=10)
    if kind == "settled":
        return dict(kind="settled", n=_log(rng, 1000, 200_000), s=1.0, precision="mixed", theta=0.0, steps=4)
    if kind == "encounter":
        return dict(kind="encounter", n=_log(rng, 1000, 98_720), s=1.0, sigma=0.06, precision="mixed", theta=0.0, steps=10)
    if kind == "batch":
        return dict(kind="batch", piles=_log(rng, 4, 256), median=_log(rng, 800, 3000), s=1.0, sigma=0.06, precision="mixed",
                    steps=10)
    if kind == "request":
        return dict(kind="request", n=_log(rng, 8000, 1_048_576), s=1.0, precision="mixed", steps=100)
    return dict(kind="field", n=_log(rng, 300, 131_072), s=5.0)


# ---------------------------------------------------------------------------------------------- inputs
def _rotations(g, n):
    q = g.standard_normal((n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)


def _mass(pile):
    return pile["density"] * 4.0 / 3.0 * math.pi * pile["radius"] ** 3


def _law(pile, *, v_max, r_med, eps, overlap_frac, G=G_SI):
    """Contact constants for restitution 0.5, sliding 0.5, rolling 0.1: the overlap at v_max is overlap_frac x r_med,
    the step a fiftieth of the contact time."""
    mu = 0.5 * float(_mass(pile).sum()) / len(pile["counts"])
    kn = mu * v_max ** 2 / (overlap_frac * r_med) ** 2
    kt = 2.0 / 7.0 * kn
    ln = math.log(2.0)
    zeta = ln / math.sqrt(math.pi ** 2 + ln ** 2)
    tc = math.pi / (math.sqrt(kn / mu) * math.sqrt(1.0 - zeta * zeta))
    return dict(G=G, dt=tc / 50, kn=kn, kt=kt, cn=2 * zeta * math.sqrt(mu * kn), ct=2 * zeta * math.sqrt(mu * kt), mu_s=0.5,
                mu_r=0.1, mu_t=0.0, w0=1e-2 * v_max / r_med, eps=eps, max_contacts=16)


def _escape(pile):
    """sqrt(2 G M / R): the speed scale of a bound pile or a collapsing cloud."""
    m = _mass(pile)
    c = (m[:, None] * pile["pos"]).sum(0) / m.sum()
    return math.sqrt(2 * G_SI * m.sum() / np.linalg.norm(pile["pos"] - c, axis=1).max())


def _cloud(g, n, mix, s, sigma, spacing):
    """n spheres in aggregates of the mix (topped up with single spheres), radii lognormal per aggregate, random
    orientations, on a jittered lattice clipped to a ball (spacing x the largest bounding diameter).  The sequence of
    grain shapes belongs to the case, everything else to the seed."""
    names = MIXES[mix]
    size = np.array([len(SHAPES[k]) for k in names] + [1])
    kind = np.random.default_rng(n).integers(0, len(names), n // int(size[:-1].min()) + 8)
    kind = kind[:int(np.searchsorted(np.cumsum(size[kind]), n, side="right"))]
    kind = np.concatenate([kind, np.full(n - int(size[kind].sum()), len(names))])
    A = len(kind)
    offs = np.zeros((len(names) + 1, 8, 3))
    bound = np.ones(len(names) + 1)
    for k, name in enumerate(names):
        offs[k, :size[k]] = SHAPES[name]
        bound[k] = 1.0 + np.linalg.norm(SHAPES[name], axis=1).max()
    sizes = s * np.exp(sigma * np.clip(g.standard_normal(A), -3, 3))
    bmax = float((bound[kind] * sizes).max())
    a = 2.0 * bmax * spacing
    m = int(math.ceil((3.0 * A / (4.0 * math.pi)) ** (1.0 / 3.0))) + 1
    ax = np.arange(-m, m + 1)
    pts = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3).astype(float)
    pts = pts[np.argsort((pts ** 2).sum(1), kind="stable")][:A]
    pts = g.permutation(pts) * a + g.uniform(-1, 1, (A, 3)) * (0.5 * a - bmax)
    counts = size[kind].astype(np.int32)
    of = np.repeat(np.arange(A), counts)
    slot = np.arange(n) - np.repeat(np.cumsum(counts) - counts, counts)
    rot = _rotations(g, A)
    pos = pts[of] + np.einsum("nij,nj->ni", rot[of], offs[kind[of], slot] * sizes[of, None])
    pile = dict(counts=counts, pos=pos, radius=sizes[of], density=np.full(n, 2500.0))
    return _stirred(g, pile, s, 0.1)


def _fcc(n, s, axes, overlap):
    """n equal spheres on an FCC packing clipped to an ellipsoid, neighbours overlapping by overlap x s, cut into
    aggregates of 1 to 8 touching spheres (runs of a random length along pairs of lattice cells).  The packing and its
    cuts belong to the case; the seed's part is how the aggregates move."""
    cell = 2.0 * s * (1.0 - overlap / 2.0) * math.sqrt(2.0)     # cubic cell edge: neighbours are edge / sqrt(2) apart
    pairs = -(-n // 8)
    ax = np.asarray(axes, float)
    c = (pairs * 2.0 / (4.0 / 3.0 * math.pi * ax.prod())) ** (1.0 / 3.0)
    m = [int(math.ceil(x * c)) + 2 for x in ax]
    g3 = np.stack(np.meshgrid(np.arange(-m[0] // 2 - 1, m[0] // 2 + 2) * 2, np.arange(-m[1], m[1] + 1),
                              np.arange(-m[2], m[2] + 1), indexing="ij"), -1).reshape(-1, 3).astype(float)
    g3 = g3[np.argsort((((g3 + [1.0, 0.5, 0.5]) / ax) ** 2).sum(1), kind="stable")][:pairs]
    basis = np.array([(0, 0, 0), (0, .5, .5), (.5, .5, 0), (.5, 0, .5), (1, 0, 0), (1.5, .5, 0), (1, .5, .5), (1.5, 0, .5)])
    pos = ((g3[:, None, :] + basis[None]) * cell).reshape(-1, 3)[:n]
    cut = np.random.default_rng(n).random(n) < 0.2                      # an aggregate starts here (mean run a few spheres)
    cut[::8] = True                              # and at every new pair of cells
    start = np.flatnonzero(cut)
    counts = np.diff(np.append(start, n)).astype(np.int32)
    return dict(counts=counts, pos=pos, radius=np.full(n, s), density=np.full(n, 2500.0))


def _stirred(g, pile, s, f):
    """Random velocities and spins, f x the pile's escape speed."""
    A = len(pile["counts"])
    v = f * _escape(pile)
    pile["vel"] = v * g.standard_normal((A, 3))
    pile["omega"] = v / s * g.standard_normal((A, 3))
    return pile


def _flyby(g, pile):
    """An Earth-mass point on a hyperbola past the pile (at rest at the origin), ten Roche distances out on the way in."""
    q, vinf = g.uniform(1.5, 4.0) * EARTH_RADIUS, g.uniform(1e3, 1e4)
    r0 = 10 * 1.26 * EARTH_RADIUS * (5514.0 / 1500.0) ** (1.0 / 3.0)
    mu = G_SI * EARTH_MASS
    a = -mu / vinf ** 2
    e = 1.0 - q / a
    p = a * (1 - e * e)
    f = -math.acos(max(-1.0, min(1.0, (p / r0 - 1.0) / e)))
    r, h = p / (1 + e * math.cos(f)), math.sqrt(mu * p)
    com = (_mass(pile)[:, None] * pile["pos"]).sum(0) / _mass(pile).sum()
    return dict(ext_mass=EARTH_MASS, ext_pos=tuple(com - np.array([r * math.cos(f), r * math.sin(f), 0.0])),
                ext_vel=(mu / h * math.sin(f), -mu / h * (e + math.cos(f)), 0.0))


def _make(case, seed):
    """The case's piles: a list of (pile, law constants)."""
    g = np.random.default_rng([seed & 0x7FFFFFFF, 20231])
    kind, s = case["kind"], case["s"]
    if kind == "cloud":
        pile = _cloud(g, case["n"], case["mix"], s, case["sigma"], case["spacing"])
        return [(pile, _law(pile, v_max=_escape(pile), r_med=s, eps=0.1 * s, overlap_frac=0.01))]
    if kind == "settled":
        pile = _stirred(g, _fcc(case["n"], s, (3.0, 2.0, 1.5), 1e-5), s, 1e-3)
        law = _law(pile, v_max=_escape(pile), r_med=s, eps=0.1 * s, overlap_frac=0.01)
        return [(pile, dict(law, spin_inc=(0.0, 0.0, 1e-9)))]
    if kind == "encounter":
        pile = _cloud(g, case["n"], "tetra", s, case["sigma"], 1.0)
        law = _law(pile, v_max=_escape(pile), r_med=s, eps=0.1 * s, overlap_frac=0.01)
        return [(pile, dict(law, **_flyby(g, pile)))]
    if kind == "batch":
        out = []
        for t in np.random.default_rng(case["piles"]).standard_normal(case["piles"]):
            n = int(min(20_000, max(500, case["median"] * math.exp(0.92 * t))))
            pile = _cloud(g, n - n % 4, "tetra", s, case["sigma"], 1.0)
            out.append((pile, _law(pile, v_max=_escape(pile), r_med=s, eps=0.1 * s, overlap_frac=0.01)))
        return out
    if kind == "request":
        pile = _fcc(case["n"], s, (1.0, 1.0, 1.0), 0.005)
        A = len(pile["counts"])
        pile["vel"], pile["omega"] = 1e-3 * g.standard_normal((A, 3)), 1e-3 / s * g.standard_normal((A, 3))
        return [(pile, _law(pile, v_max=1e-2, r_med=s, eps=0.1 * s, overlap_frac=0.02, G=0.0))]
    raise ValueError(kind)


def _field(case, seed):
    """Spheres of a collapse cloud as a host program holds them: FP32 positions and masses, contiguous aggregates."""
    g = np.random.default_rng([seed & 0x7FFFFFFF, 977])
    pile = _cloud(g, case["n"], "simple", case["s"], 0.2, 2.5)
    m = _mass(pile)
    pm = np.concatenate([pile["pos"], m[:, None]], 1).astype(np.float32)
    return pm, m, np.repeat(np.arange(len(pile["counts"]), dtype=np.int32), pile["counts"])


# ---------------------------------------------------------------------------------------------- one pass
_FIELDS = ("COM", "VEL", "QUAT", "OMEGA", "ACC")
_CONTACT_FIELDS = _FIELDS + ("TORQUE_STORED",)
_KEPT = ("COM", "QUAT")      # FP64 also in the mixed path (48-bit state); the rest follows from FP32 forces


def _fields(case):
    return _CONTACT_FIELDS if case["kind"] in ("settled", "request") else _FIELDS


def _add(world, pile, law, precision):
    from paper_2311_11322_gb300 import workloads as W
    ic = W.PileIC(counts=pile["counts"], pos=pile["pos"], radius=pile["radius"], density=pile["density"], vel=pile["vel"],
                  omega=pile["omega"])
    p = W.Params(**law).replace(precision=W.PRECISION_FP64 if precision == "fp64" else W.PRECISION_MIXED)
    return world.add_pile(ic, p)


def prepare(case, seed):
    from paper_2311_11322_gb300 import dem
    if case["kind"] == "field":
        pm, m, agg = _field(case, seed)
        return dict(case=case, call=dem.load().dem_gravity_noalloc, pm=torch.from_numpy(pm).cuda(),
                    m=torch.from_numpy(m).cuda(), agg=torch.from_numpy(agg).cuda(),
                    out=torch.zeros(len(m), 4, dtype=torch.float64, device="cuda"))
    world = dem.World()
    state = dict(case=case, world=world, piles=_make(case, seed))
    if case["kind"] != "request":
        if case.get("theta"):
            world.set_tuning("grav_theta", case["theta"])
        state["ids"] = [_add(world, pile, law, case["precision"]) for pile, law in state["piles"]]
    A = sum(len(pile["counts"]) for pile, _ in state["piles"])
    # the driver's own result arrays, filled by every read
    state["out"] = {f: np.zeros((A, 4 if f == "QUAT" else 3)) for f in _fields(case)}
    return state


def _read(state, ids):
    out, a0 = state["out"], 0
    for pid in ids:
        a1 = a0 + state["world"].piles[pid][0]
        for f, x in out.items():
            state["world"].read(pid, f, out=x[a0:a1])
        a0 = a1
    mixed = state["case"]["precision"] == "mixed"
    return {f: x.astype(np.float32) if mixed and f not in _KEPT else x for f, x in out.items()}


def run(state):
    case = state["case"]
    if case["kind"] == "field":
        st = torch.cuda.current_stream().cuda_stream
        rc = state["call"](state["pm"].data_ptr(), ctypes.c_void_p(state["m"].data_ptr()), state["agg"].data_ptr(),
                           case["n"], G_SI, 0.1 * case["s"], ctypes.c_void_p(state["out"].data_ptr()), st, None, 0)
        if rc != 0:
            raise RuntimeError(f"dem_gravity_noalloc: status {rc}")
        return state["out"][:, :3].float()   # pair terms are FP32
    world = state["world"]
    if case["kind"] == "request":
        (pile, law), = state["piles"]
        pid = _add(world, pile, law, case["precision"])
        world.step(case["steps"])
        out = _read(state, [pid])
        world.remove(pid)
        return out
    world.step(case["steps"])
    return _read(state, state["ids"])


# ---------------------------------------------------------------------------------------------- work of a pass
def work(case):
    """Pairs of gravity (27 flop per unordered pair of the direct sum; about 2,500 interactions of 120 flop per sphere for
    the tree), about 200 flop per touching pair, and the state and contact records read and written once a step."""
    kind = case["kind"]
    if kind == "field":
        n = case["n"]
        return dict(bytes=28.0 * n + 24.0 * n, flops=13.5 * n * n)
    if kind == "batch":
        ns = [case["median"] * 1.4] * case["piles"]      # about the mean of the sizes drawn
        pairs = 0.5 * case["piles"] * (1.9 * case["median"]) ** 2
    else:
        ns = [case["n"]]
        pairs = 0.0 if kind == "request" else 0.5 * case["n"] ** 2
    n = float(sum(ns))
    contacts = {"settled": 4.7, "request": 4.7}.get(kind, 0.0) * n
    grav = 2500.0 * 120.0 * n if case.get("theta") else 27.0 * pairs
    scale = 2.0 if case["precision"] == "fp64" else 1.0
    step_bytes = scale * (84.0 * n + 32.0 * contacts) + 400.0 * n / 3.5
    return dict(bytes=case["steps"] * step_bytes + 128.0 * n / 3.5, flops=case["steps"] * (grav + 200.0 * contacts))


# ---------------------------------------------------------------------------------------------- 64-bit reference
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=_dev())


def _quat_R(q):
    w, x, y, z = q.T
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _mv(M, v):
    return (M @ v.unsqueeze(-1)).squeeze(-1)


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _rhs(q, w, I, Iinv):
    p = torch.cat([torch.zeros_like(w[:, :1]), w], 1)
    a0, a1, a2, a3 = q.T
    b0, b1, b2, b3 = p.T
    dq = 0.5 * torch.stack([a0 * b0 - a1 * b1 - a2 * b2 - a3 * b3, a0 * b1 + a1 * b0 + a2 * b3 - a3 * b2,
                            a0 * b2 - a1 * b3 + a2 * b0 + a3 * b1, a0 * b3 + a1 * b2 - a2 * b1 + a3 * b0], 1)
    return dq, _mv(Iinv, -_cross(w, _mv(I, w)))


def _rotate(q, w, I, Iinv, h):
    k1 = _rhs(q, w, I, Iinv)
    k2 = _rhs(q + 0.5 * h * k1[0], w + 0.5 * h * k1[1], I, Iinv)
    k3 = _rhs(q + 0.5 * h * k2[0], w + 0.5 * h * k2[1], I, Iinv)
    k4 = _rhs(q + h * k3[0], w + h * k3[1], I, Iinv)
    q = q + h / 6.0 * (k1[0] + 2 * k2[0] + 2 * k3[0] + k4[0])
    w = w + h / 6.0 * (k1[1] + 2 * k2[1] + 2 * k3[1] + k4[1])
    return q / q.norm(dim=1, keepdim=True), w


def _close_pairs(x, s, agg, reach):
    """Pairs (i < j) of different aggregates whose centres are nearer than the radii sum plus reach."""
    cell = 2.0 * float(s.max()) + reach
    c = torch.floor((x - x.min(0).values) / cell).long() + 1
    dim = c.max(0).values + 2
    key = (c[:, 0] * dim[1] + c[:, 1]) * dim[2] + c[:, 2]
    order = torch.argsort(key, stable=True)
    sk = key[order]
    found = []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                k2 = key + (dx * dim[1] + dy) * dim[2] + dz
                lo = torch.searchsorted(sk, k2)
                cnt = torch.searchsorted(sk, k2, right=True) - lo
                i = torch.repeat_interleave(torch.arange(len(x), device=x.device), cnt)
                j = order[torch.repeat_interleave(lo - (cnt.cumsum(0) - cnt), cnt) + torch.arange(len(i), device=x.device)]
                keep = (i < j) & (agg[i] != agg[j]) & ((x[i] - x[j]).norm(dim=1) < s[i] + s[j] + reach)
                found.append(torch.stack([i[keep], j[keep]]))
    return torch.cat(found, 1)


def _gravity(x, m, agg, eps, G):
    """F_i = G m_i sum_j m_j (r_j - r_i) / (|r_j - r_i|^2 + eps^2)^1.5 over spheres of other aggregates."""
    F = torch.zeros_like(x)
    n = len(x)
    step = max(1, min(n, 60_000_000 // n))
    for b in range(0, n, step):
        d = [x[None, :, c] - x[b:b + step, None, c] for c in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2]).add_(eps * eps)
        w = m[None, :] / (r2 * r2.sqrt())
        w.masked_fill_(agg[None, :] == agg[b:b + step, None], 0.0)
        for c in range(3):
            F[b:b + step, c] = (d[c] * w).sum(1)
    return G * m[:, None] * F


def _simulate(pile, law, steps):
    """The whole step in 64 bits: kick and drift, torque-free RK4 rotation, contacts, gravity, planet, closing kick."""
    h, G = law["dt"], law["G"]
    dev = _dev()
    counts = torch.as_tensor(pile["counts"], dtype=torch.long, device=dev)
    A = len(counts)
    agg = torch.repeat_interleave(torch.arange(A, device=dev), counts)
    x, s, m = _t(pile["pos"]), _t(pile["radius"]), _t(_mass(pile))

    def total(v):
        return torch.zeros((A,) + v.shape[1:], dtype=torch.float64, device=dev).index_add_(0, agg, v)

    first = x[counts.cumsum(0) - counts]
    M = total(m)
    r = first + total(m[:, None] * (x - first[agg])) / M[:, None]
    b = x - r[agg]
    eye = torch.eye(3, dtype=torch.float64, device=dev)
    I = total((0.4 * m * s * s + m * (b * b).sum(1))[:, None, None] * eye - m[:, None, None] * b[:, :, None] * b[:, None, :])
    Iinv = torch.linalg.inv(I)
    v, wb = _t(pile["vel"]), _t(pile["omega"])
    q = torch.zeros(A, 4, dtype=torch.float64, device=dev)
    q[:, 0] = 1.0
    acc, N = torch.zeros_like(v), torch.zeros_like(v)
    mp = law.get("ext_mass", 0.0)
    P, PV, PA = (_t(law.get("ext_pos", (0, 0, 0))), _t(law.get("ext_vel", (0, 0, 0))), _t((0, 0, 0)))
    spin = _t(law.get("spin_inc", (0, 0, 0)))
    i, j = _close_pairs(x, s, agg, 0.2 * float(s.max()))
    hist = torch.zeros(len(i), 3, dtype=torch.float64, device=dev)
    for _ in range(steps):
        R = _quat_R(q)
        v = v + 0.5 * h * acc
        wb = wb + 0.5 * h * _mv(Iinv, _mv(R.mT, N))
        r = r + h * v
        q, wb = _rotate(q, wb, I, Iinv, h)
        R = _quat_R(q)
        ws = _mv(R, wb + 0.5 * h * _mv(Iinv, _mv(R.mT, N)))
        lever = _mv(R[agg], b)
        x = r[agg] + lever
        w = ws[agg]
        u = (v + 0.5 * h * acc)[agg] + _cross(w, lever)
        F, T = torch.zeros_like(x), torch.zeros_like(x)
        if len(i):
            f, ta, tb, hist = _contacts(x, u, w, s, i, j, hist, law)
            F.index_add_(0, i, f).index_add_(0, j, -f)
            T.index_add_(0, i, ta).index_add_(0, j, tb)
        if G:
            F += _gravity(x, m, agg, law["eps"], G)
        if mp:
            PV = PV + 0.5 * h * PA
            P = P + h * PV
            d = P - x
            fe = (G * mp * m / (d * d).sum(1) ** 1.5)[:, None] * d
            F += fe
            PA = -fe.sum(0) / mp
            PV = PV + 0.5 * h * PA
        N = total(_cross(lever, F) + T)
        acc = total(F) / M[:, None]
        rc = (M[:, None] * r).sum(0) / M.sum()
        v = v + 0.5 * h * acc + _cross(spin.expand_as(r), r - rc)
        wb = wb + 0.5 * h * _mv(Iinv, _mv(R.mT, N)) + _mv(R.mT, spin.expand_as(r))
    return dict(COM=r, VEL=v, QUAT=q, OMEGA=_mv(R, wb), ACC=acc, TORQUE_STORED=N)


def _contacts(x, u, w, s, i, j, hist, law):
    """Forces on i (and minus that on j), torques on both about their centres, and the tangential displacement kept
    while a pair touches."""
    kn, kt, cn, ct, h = law["kn"], law["kt"], law["cn"], law["ct"], law["dt"]
    dot = lambda a, b: (a * b).sum(1, keepdim=True)  # noqa: E731
    d = x[j] - x[i]
    dist = d.norm(dim=1, keepdim=True)
    si, sj = s[i, None], s[j, None]
    over = si + sj - dist
    n = d / dist
    la = 0.5 * dist + 0.5 * (si - sj) * (si + sj) / dist
    lb = dist - la
    rel = (u[j] + _cross(w[j], -lb * n)) - (u[i] + _cross(w[i], la * n))
    un = dot(rel, n)
    ut = rel - un * n
    fn = cn * un - kn * over
    Sp = hist - dot(hist, n) * n
    Spm = Sp.norm(dim=1, keepdim=True)
    Sp = torch.where(Spm > 0, Sp * (hist.norm(dim=1, keepdim=True) / Spm.clamp_min(1e-300)), torch.zeros_like(Sp))
    S = Sp + h * ut
    FT = kt * S + ct * ut
    FTm, cap = FT.norm(dim=1, keepdim=True), law["mu_s"] * fn.abs()
    slip = FTm > cap
    FT = torch.where(slip, FT * (cap / FTm.clamp_min(1e-300)), FT)
    S = torch.where(slip, (FT - ct * ut) / kt, S)
    wr = w[i] - w[j]
    wr = wr - dot(wr, n) * n
    Mr = -law["mu_r"] * fn.abs() * (si * sj / (si + sj)) * wr / wr.norm(dim=1, keepdim=True).clamp_min(law["w0"])
    F = fn * n + FT
    hit = (over > 0).double()
    return hit * F, hit * (_cross(la * n, F) + Mr), hit * (_cross(lb * n, F) - Mr), hit * S


def exact(case, seed):
    """What run() returns for a fresh state, in 64 bits."""
    if case["kind"] == "field":
        pm, m, agg = _field(case, seed)
        pm = _t(pm)
        # the call's own arguments: FP32 positions and pair masses, FP64 masses in the outer factor
        F = _gravity(pm[:, :3], pm[:, 3], torch.as_tensor(agg, device=_dev()), 0.1 * case["s"], G_SI)
        return (F * (_t(m) / pm[:, 3])[:, None]).cpu().numpy()
    got = [_simulate(pile, law, case["steps"]) for pile, law in _make(case, seed)]
    return {f: torch.cat([g[f] for g in got]).cpu().numpy() for f in _fields(case)}
