"""NSBC settings past the range of float, which lbm_set_nsbc accepts: a uniform state
equal to the far field stays as it is on every storage."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("gamma,beta", [(1e39, 0.0), (-1e39, 0.5), (0.6, 1e39), (0.6, -1e300)])
@pytest.mark.parametrize("order", [1, 2])
def test_far_field_stays(lbm, storage, gamma, beta, order):
    one, zero = np.ones((20, 30)), np.zeros((20, 30))
    with lbm.Simulation(30, 20, 0.6, storage=storage, gamma=gamma, beta=beta, grad_order=order) as s:
        first = s.init(one, zero, zero).populations()
        assert np.array_equal(s.step(5).populations(), first)
        assert np.array_equal(s.step(64).populations(), first)
