"""A wait of a resident domain's blocks that runs out: every call that waits for the
stream says so, and a new state starts clean."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


def _fields(n):
    rng = np.random.default_rng(n)
    return [b + 1e-3 * rng.standard_normal((n, n)) for b in (1.0, 0.0, 0.0)]


def _timeout(lbm, call):
    with pytest.raises(lbm.LbmError) as e:
        call()
    assert e.value.code == lbm.LBM_ETIMEOUT


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("again", ["init", "populations", "load_state"])
def test_given_up_wait_is_reported_until_a_new_state(lbm, storage, again):
    n = 300
    f = _fields(n)
    with lbm.Simulation(n, n, 0.6, storage=storage) as s:
        s.init(*f)
        pop = s.populations()
        record, _ = lbm.lbm_save_state(s.h)

        def new_state():
            if again == "init":
                s.init(*f)
            elif again == "populations":
                s.set_populations(pop)
            else:
                lbm.lbm_load_state(s.h, record)

        new_state()
        ref = s.step(128).populations()
        s.init(*f)
        lbm.lbm_set_wait_limit(s.h, 0)
        s.step(64)
        s.step(64)
        for call in (s.status, s.macros, s.populations, s.reduce, lambda: lbm.lbm_save_state(s.h),
                     lambda: lbm.lbm_reduce_noalloc(s.h)):
            _timeout(lbm, call)
        lbm.lbm_set_wait_limit(s.h, 2_000_000_000)
        s.step(1)
        _timeout(lbm, s.macros)  # a later good step does not make the state one
        new_state()
        s.status()
        assert np.array_equal(s.step(128).populations(), ref)
        s.reduce()


def test_limit_range_and_selftest(lbm):
    with lbm.Simulation(8, 8, 0.6) as s:
        for bad in (-1, 4_000_000_001):
            with pytest.raises(lbm.LbmError):
                lbm.lbm_set_wait_limit(s.h, bad)
    assert lbm.lbm_wait_selftest(100_000) == lbm.LBM_ETIMEOUT
