"""A domain kept on chip for a call's steps (resident tiles) is bit-identical to the
kernel pair: one tile and many, ragged sizes up to the largest that fit, every
storage, edge kind, order and corner reading, and step counts on both sides of
the shortest resident launch and of its rounds."""
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


@pytest.mark.parametrize("nx,ny", [(8, 8), (17, 200), (128, 128), (200, 201), (401, 399), (613, 377), (640, 640)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "f64"])
@pytest.mark.parametrize("model,edges,far,order,corner", [
    ("bgk", NSBC, (0.0, 0.0), 1, 0), ("mrt", VELOCITY, (0.05, 0.01), 2, 1), ("mrt", CHANNEL, (0.05, 0.0), 1, 0),
    ("bgk", PERIODIC, (0.0, 0.0), 1, 0)])
def test_resident_equals_pair(lbm, nx, ny, storage, model, edges, far, order, corner):
    rng = np.random.default_rng(nx + ny)
    f = [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, far[0], far[1])]
    out = []
    for pair in (True, False):
        with lbm.Simulation(nx, ny, 0.6, storage=storage, mrt_rates=(1.4, 1.4, 1.2), farfield_u=far, collision=model,
                            edges=edges, grad_order=order, corner_mode=corner, beta=0.1) as s:
            s.init(*f)
            if pair:
                s.set_launch(128, 1, 0)
            for n in (64, 70, 63, 5):
                s.step(n)
            s.status()
            out.append(s.populations())
    assert np.array_equal(out[0], out[1])
