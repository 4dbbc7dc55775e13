"""Each launch form, asked for and known to have run, against the kernel pair bit by
bit: tiles on every storage (double among them), resident domains, and the form
lbm_step picks by itself, which lbm_get_form names."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

NSBC = ["nsbc"] * 4
VELOCITY = [("velocity", 0.03, 0.01), "nsbc", "nsbc", ("velocity", 0.0, -0.02)]
CHANNEL = [("velocity", 0.05, 0.0), "nsbc", "periodic", "periodic"]
PERIODIC = ["periodic"] * 4
SETTINGS = [("bgk", NSBC, (0.0, 0.0), 1, 0), ("mrt", VELOCITY, (0.05, 0.01), 2, 1), ("mrt", CHANNEL, (0.05, 0.0), 1, 0),
            ("bgk", PERIODIC, (0.0, 0.0), 1, 0)]


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


def _runs(lbm, nx, ny, storage, setting, choose, steps):
    """Populations of the kernel pair and of the form `choose` asks for, and that form."""
    model, edges, far, order, corner = setting
    rng = np.random.default_rng(nx + ny)
    f = [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, far[0], far[1])]
    out = []
    for pair in (True, False):
        with lbm.Simulation(nx, ny, 0.6, storage=storage, mrt_rates=(1.4, 1.4, 1.2), farfield_u=far, collision=model,
                            edges=edges, grad_order=order, corner_mode=corner, beta=0.1) as s:
            s.init(*f)
            if pair:
                s.set_launch(128, 1, 0)
            else:
                choose(s)
            form = s.form
            for n in steps:
                s.step(n)
            s.status()
            out.append(s.populations())
    return out[0], out[1], form


@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 13), (64, 40), (131, 75), (257, 9), (200, 201)])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("setting", SETTINGS)
def test_tiles_equal_pair(lbm, nx, ny, storage, setting):
    ref, got, form = _runs(lbm, nx, ny, storage, setting, lambda s: s.set_tiles(), (1, 2, 3, 7, 16, 29))
    assert form[0] == "tiles" and form[1] >= 1
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("nx,ny", [(8, 8), (17, 200), (128, 128), (401, 399), (500, 610)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("setting", SETTINGS)
def test_resident_tiles_equal_pair(lbm, nx, ny, storage, setting):
    ref, got, form = _runs(lbm, nx, ny, storage, setting, lambda s: s.set_tiles(), (64, 70, 63, 5))
    assert form[0] == "tiles" and form[2] == 64
    assert np.array_equal(got, ref)


def test_tiles_refused(lbm):
    for nx, ny in ((7, 9), (9, 7), (2048, 1025), (65536, 32)):
        with lbm.Simulation(nx, ny, 0.6) as s:
            with pytest.raises(lbm.LbmError):
                s.set_tiles()


def test_form_follows_the_setters(lbm):
    with lbm.Simulation(300, 300, 0.6) as s:
        for choose, form, per in ((lambda: s.set_launch(128, 1, 0), "pair", 1), (s.set_fused, "fused", 1),
                                  (lambda: s.set_staged(3), "staged", 1), (s.set_twostep, "pass", 4),
                                  (lambda: s.set_twostep(False), "pair", 1)):
            choose()
            assert s.form == (form, per, 0)


def test_forms_in_bounds():
    """No form of several steps makes an access that the bounds-checked build rejects."""
    from paper_2005_08674_gb300 import build
    build.build(check=True)
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked_forms.py")], capture_output=True, text=True,
                       timeout=900, env=dict(os.environ, LBM_CHECKED="1"))
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["checked"] and out["rejected"] == 0, out


CASES = [
    # open squares, one and two periodic axes
    (128, 128, "f32", "bgk", NSBC, "tiles", True), (300, 300, "f32", "mrt", NSBC, "tiles", True),
    (300, 300, "f16", "bgk", NSBC, "fused", True), (128, 128, "f32", "mrt", CHANNEL, "tiles", True),
    (300, 300, "f32", "bgk", CHANNEL, "fused", False), (64, 64, "f32", "bgk", PERIODIC, "fused", True),
    (300, 300, "f32", "bgk", PERIODIC, "fused", False), (500, 500, "f16", "bgk", PERIODIC, "fused", False),
    (500, 500, "f32", "bgk", NSBC, "fused", True), (500, 500, "f32", "mrt", NSBC, "fused", False),
    (200, 200, "f64", "bgk", NSBC, "fused", False),
    # wide ones of few rows and their transposes
    (13000, 8, "f32", "bgk", NSBC, "fused", True), (13000, 8, "f32", "mrt", NSBC, "fused", False),
    (13000, 8, "f16", "bgk", CHANNEL, "fused", False), (8, 13000, "f32", "bgk", NSBC, "tiles", True),
    (8, 13000, "f16", "bgk", NSBC, "tiles", True), (3, 3, "f32", "bgk", NSBC, "fused", False),
    (65536, 20, "f32", "bgk", NSBC, "pair", False), (20, 65536, "f32", "bgk", NSBC, "pass", False),
    (65536, 48, "f16", "bgk", NSBC, "pair", False), (48, 65536, "f16", "bgk", NSBC, "pass", False),
    (20000, 100, "f32", "bgk", NSBC, "pass", False), (4, 40000, "f32", "bgk", NSBC, "pair", False),
    # large ones
    (1024, 1024, "f32", "bgk", NSBC, "pair", False), (1201, 1003, "f32", "bgk", NSBC, "pass", False),
    (1801, 1600, "f16", "bgk", NSBC, "pass", False), (1500, 1500, "f32", "bgk", CHANNEL, "pair", False)]


@pytest.mark.parametrize("nx,ny,storage,model,edges,form,resident", CASES)
def test_picked_form(lbm, nx, ny, storage, model, edges, form, resident):
    """The form lbm_step picks by itself: each one where it is the faster."""
    with lbm.Simulation(nx, ny, 0.6, storage=storage, collision=model, edges=edges) as s:
        assert s.form[0] == form and (s.form[2] > 0) == resident


@pytest.mark.parametrize("bx", [64, 128, 256, 512])
@pytest.mark.parametrize("nx,ny", [(3, 3), (5, 7), (257, 9), (131, 75), (517, 40)])
def test_pair_with_and_without_prefetch(lbm, nx, ny, bx):
    """f32 at rest: the bulk kernel that holds no prefetch against the one that does."""
    out = []
    for pf in (0, 1):
        ref, got, form = _runs(lbm, nx, ny, "f32", SETTINGS[0], lambda s: s.set_launch(bx, 2, pf), (1, 16))
        assert form[0] == "pair"
        out += [ref, got]
    assert all(np.array_equal(out[0], a) for a in out[1:])


@pytest.mark.parametrize("nx,ny,storage,setting", [(300, 300, "f16", SETTINGS[0]), (1000, 30, "f32", SETTINGS[0]),
                                                   (43, 301, "f16", SETTINGS[3]), (200, 201, "bf16", SETTINGS[2])])
def test_left_over_steps_as_tiles(lbm, nx, ny, storage, setting):
    """What the graphs of the one-launch form leave: tiles from three steps on, the same bits."""
    def choose(s):
        lbm.lbm_profile(s.h, True)

    def launches(s, n):
        s.step(n)
        return lbm.lbm_profile_read(s.h)[1]
    ref, got, form = _runs(lbm, nx, ny, storage, setting, choose, (1, 3, 4, 5, 15, 16, 20, 31, 4))
    assert form[0] == "fused"
    assert np.array_equal(got, ref)
    ref, got, _ = _runs(lbm, nx, ny, storage, setting, lambda s: None, (1, 3, 4, 5, 15, 16, 20, 31, 4))
    assert np.array_equal(got, ref)
    model, edges, far, order, corner = setting
    with lbm.Simulation(nx, ny, 0.6, storage=storage, mrt_rates=(1.4, 1.4, 1.2), farfield_u=far, collision=model,
                        edges=edges, grad_order=order, corner_mode=corner) as s:
        s.init(*[np.full((ny, nx), b) for b in (1.0, far[0], far[1])])
        lbm.lbm_profile(s.h, True)
        assert launches(s, 2) == 2
        assert launches(s, 3) < 3
        assert launches(s, 15) < 15
        assert 16 < launches(s, 20) < 20
