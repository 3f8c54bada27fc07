"""GPU: state reads on either side of the size at which they change route (fewer than 32,768 values are formed in the
world's pinned staging buffer, more in the pile's per-step records and copied), and what they leave behind."""
import numpy as np
import pytest

from paper_2311_11322_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STATE = ("COM", "VEL", "QUAT", "OMEGA_BODY", "ACC", "TORQUE_STORED")


@pytest.fixture(scope="module")
def dem():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2311_11322_gb300 import dem as D
    return D


def pile(n_agg, precision):
    """n_agg dumbbells with self-gravity, all spinning."""
    rng = np.random.default_rng(n_agg)
    box = 6.0 * n_agg ** (1.0 / 3.0)
    com = np.repeat(rng.uniform(-box, box, (n_agg, 3)), 2, axis=0)
    com[0::2, 0] += 0.5
    com[1::2, 0] -= 0.5
    ic = W.PileIC(counts=np.full(n_agg, 2, np.int32), pos=com, radius=np.full(2 * n_agg, 0.5),
                  density=np.full(2 * n_agg, 2500.0), vel=rng.standard_normal((n_agg, 3)),
                  omega=rng.standard_normal((n_agg, 3)))
    return ic, W.Params(G=6.67430e-11, dt=1e-3, kn=1e3, eps=0.1, precision=precision)


# 3 n_agg and 4 n_agg below, at and above 32,768
@pytest.mark.parametrize("n_agg", [1, 8191, 8192, 10922, 10923])
@pytest.mark.parametrize("precision", [W.PRECISION_MIXED, W.PRECISION_FP64])
def test_reads_on_both_routes(dem, n_agg, precision):
    ic, p = pile(n_agg, precision)
    other = pile(40, precision)
    with dem.World() as w:      # unread until the end
        w.add_pile(*other)
        pid = w.add_pile(ic, p)
        w.step(4)
        ref = {f: w.read(pid, f) for f in STATE}
    with dem.World() as w:
        small = w.add_pile(*other)
        pid = w.add_pile(ic, p)
        for _ in range(4):
            w.step(1)
            # the asynchronous read takes a route of its own
            for f in STATE:
                out = np.full((n_agg, 4 if f == "QUAT" else 3), np.nan)
                w.read_async(pid, f, out)
                w.read_wait()
                assert np.array_equal(out, w.read(pid, f)), f
            w.read(small, "COM")
            q, wb, om = w.read(pid, "QUAT"), w.read(pid, "OMEGA_BODY"), w.read(pid, "OMEGA")
        v, a, t = q[:, 1:], wb, q[:, :1]     # R(q) w = w + 2 q0 (v x w) + 2 v x (v x w)
        rot = a + 2 * t * np.cross(v, a) + 2 * np.cross(v, np.cross(v, a))
        # (the same polynomial of the values read: some ten FP64 roundings on either side)
        assert np.all(np.abs(om - rot) <= 1e-14 * np.abs(wb).max())
        for f in STATE:          # and reading changed nothing
            assert np.array_equal(w.read(pid, f), ref[f]), f
