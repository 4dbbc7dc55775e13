"""lbm_profile times the launches that lbm_step makes: their number per form, and the
state they leave."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


# (size, storage, collision, steps) -> launches counted as bulk and as NSBC
@pytest.mark.parametrize("nx,ny,storage,model,steps,bulk,nsbc", [
    (300, 300, "f32", "bgk", 100, 1, 0), (300, 300, "f32", "bgk", 1, 1, 0), (400, 400, "f32", "mrt", 20, 20, 0),
    (200, 200, "f64", "bgk", 20, 20, 0), (1024, 1024, "f32", "bgk", 20, 20, 20), (1201, 1003, "f32", "bgk", 22, 6, 0),
    (1201, 1003, "f32", "bgk", 1, 1, 1)])
def test_profiled_launches(lbm, nx, ny, storage, model, steps, bulk, nsbc):
    rng = np.random.default_rng(nx)
    f = [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, 0.0, 0.0)]
    out = []
    for profile in (False, True):
        with lbm.Simulation(nx, ny, 0.6, storage=storage, collision=model) as s:
            s.init(*f)
            form = s.form
            if profile:
                lbm.lbm_profile(s.h, True)
                assert s.form == form
            s.step(steps)
            if profile:
                ms, n, nsbc_ms, n_nsbc = lbm.lbm_profile_read(s.h)
                assert (n, n_nsbc) == (bulk, nsbc) and ms > 0.0 and (nsbc_ms > 0.0) == (nsbc > 0)
                lbm.lbm_profile(s.h, False)
            out.append(s.populations())
    assert np.array_equal(*out)
