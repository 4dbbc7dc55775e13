"""Several steps per launch (tiles of a small domain, passes over a large one):
the launch form lbm_step picks by itself is bit-identical to the kernel pair --
at the edges of tiles and passes, on every storage, with NSBC, velocity and
periodic edges, both orders and corner readings, and step counts that leave
every remainder."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NSBC = ["nsbc"] * 4
VELOCITY = [("velocity", 0.03, 0.01), "nsbc", "nsbc", ("velocity", 0.0, -0.02)]
CHANNEL = [("velocity", 0.05, 0.0), "nsbc", "periodic", "periodic"]
PERIODIC = ["periodic"] * 4


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


def _run(lbm, nx, ny, storage, pair, fields, steps, **kw):
    with lbm.Simulation(nx, ny, 0.6, storage=storage, mrt_rates=(1.4, 1.4, 1.2), **kw) as s:
        s.init(*fields)
        if pair:
            s.set_launch(128, 1, 0)
        for n in steps:
            s.step(n)
        s.status()
        return s.populations()


# (nx, ny): below and above the smallest tile, ragged, a narrow strip, 300^2
# (tiles), 1201 x 1003 (passes in f32) and 1801 x 1600 (passes in 16 bits)
@pytest.mark.parametrize("nx,ny", [(7, 9), (8, 8), (9, 13), (64, 40), (131, 75), (257, 9), (300, 300), (1201, 1003),
                                   (1801, 1600)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f64"])
@pytest.mark.parametrize("model,edges,far,order,corner", [
    ("bgk", NSBC, (0.0, 0.0), 1, 0), ("mrt", VELOCITY, (0.05, 0.01), 2, 1), ("mrt", CHANNEL, (0.05, 0.0), 1, 0),
    ("bgk", PERIODIC, (0.0, 0.0), 1, 0)])
def test_picked_form_equals_pair(lbm, nx, ny, storage, model, edges, far, order, corner):
    if nx > 1000 and (storage in ("bf16", "f64") or edges is PERIODIC):
        pytest.skip("one storage of each width and the edges a pass serves")
    rng = np.random.default_rng(nx + ny)
    f = [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, far[0], far[1])]
    kw = dict(farfield_u=far, collision=model, edges=edges, grad_order=order, corner_mode=corner, beta=0.1)
    steps = (1, 2, 3, 4, 5, 17) if nx > 1000 else (1, 2, 3, 7, 16, 29)
    ref = _run(lbm, nx, ny, storage, True, f, steps, **kw)
    got = _run(lbm, nx, ny, storage, False, f, steps, **kw)
    assert np.array_equal(got, ref)


def test_batch_picks_passes(lbm):
    """An f32 batch of over a million nodes takes passes; every instance equals its single run."""
    class W:
        farfield_rho, farfield_u = 1.0, (0.0, 0.0)

        def __init__(self, nx, ny):
            self.nx, self.ny, self.tau = nx, ny, 0.6
    ws = [W(1003, 900), W(9, 8), W(400, 301), W(60, 257)]
    rng = np.random.default_rng(1)
    fields = [[b + 1e-3 * rng.standard_normal((w.ny, w.nx)) for b in (1.0, 0.0, 0.0)] for w in ws]
    with lbm.Batch(ws, storage="f32") as b:
        for k, f in enumerate(fields):
            b.init(k, *f)
        for n in (1, 2, 3, 5, 18):
            b.step(n)
        b.status()
        for k, (w, f) in enumerate(zip(ws, fields)):
            with lbm.Simulation(w.nx, w.ny, w.tau) as s:
                s.set_launch(128, 1, 0)
                ref = s.init(*f).step(29).macros()
            for a, c in zip(b.macros(k), ref):
                assert np.array_equal(a, c), (w.nx, w.ny)
