"""The counters and flags of a handle's kernels: many handles at once, more than the
library holds room for, and a slot whose last owner's wait had given up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


def _fields(nx, ny, seed):
    rng = np.random.default_rng(seed)
    return [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, 0.0, 0.0)]


def test_more_handles_than_slots(lbm):
    sims = [lbm.Simulation(64, 48, 0.6) for _ in range(70)]
    for k, s in enumerate(sims):
        s.init(*_fields(64, 48, k))
    for s in sims:
        assert s.form[2] == 64  # resident: flags and counters in use
        s.step(70)
    for k in (0, 63, 64, 69):
        with lbm.Simulation(64, 48, 0.6) as ref:
            want = ref.init(*_fields(64, 48, k)).set_launch(128, 1, 0).step(70).populations()
        assert np.array_equal(sims[k].populations(), want)
    for s in sims:
        s.status()
        s.close()


def test_slot_after_a_given_up_wait(lbm):
    f = _fields(200, 201, 1)
    for _ in range(3):
        with lbm.Simulation(200, 201, 0.6) as s:
            s.init(*f)
            lbm.lbm_set_wait_limit(s.h, 0)
            s.step(64)
            with pytest.raises(lbm.LbmError):
                s.status()
    out = []
    for pair in (True, False):
        with lbm.Simulation(200, 201, 0.6) as s:
            s.init(*f)
            if pair:
                s.set_launch(128, 1, 0)
            out.append(s.step(64).status().populations())
    assert np.array_equal(*out)


def test_handle_moved_between_streams(lbm):
    import torch
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    f = _fields(1201, 1003, 2)
    with lbm.Simulation(1201, 1003, 0.6) as s:
        want = s.init(*f).set_launch(128, 1, 0).step(80).populations()
    for _ in range(3):
        s = lbm.Simulation(1201, 1003, 0.6, stream=a)
        s.init(*f).step(40)
        b.wait_stream(a)
        lbm.lbm_set_stream(s.h, b.cuda_stream)
        s.step(40)
        assert np.array_equal(s.populations(), want)
        s.close()
