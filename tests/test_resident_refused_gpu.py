"""A stream that may not hold all blocks of a resident domain at once refuses its
cooperative launch; lbm_step and lbm_autotune then take another form.  The refusal
is an error code from a stand-in for the launch call, in a child process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = """
#include <stddef.h>
static int refused;
int cudaLaunchCooperativeKernel(const void* f, ...) { (void)f; ++refused; return %d; }
int refused_launches(void) { return refused; }
"""

CHILD = """
import ctypes, sys
import numpy as np, torch
sys.path.insert(0, {root!r})
from paper_2005_08674_gb300 import lbm
refused = ctypes.CDLL({shim!r}).refused_launches
for nx, ny, storage in ((128, 96, "f32"), (500, 400, "f16")):
    rng = np.random.default_rng(nx)
    f = [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, 0.0, 0.0)]
    out = []
    for way in ("pair", "picked", "tuned"):
        with lbm.Simulation(nx, ny, 0.6, storage=storage) as s:
            s.init(*f)
            before = refused()
            if way == "pair":
                s.set_launch(128, 1, 0)
            elif way == "tuned":
                s.autotune()
            got = s.step(100).step(65).populations()
            assert (refused() > before) == (way != "pair"), way
        out.append(got)
    assert all(np.array_equal(out[0], a) for a in out[1:]), (nx, ny)
print("same bits")
"""


@pytest.mark.parametrize("code", [720, 801])  # cudaErrorCooperativeLaunchTooLarge, cudaErrorNotSupported
def test_refused_cooperative_launch(tmp_path, code):
    from paper_2005_08674_gb300 import build
    build.build()
    src, shim = tmp_path / "shim.c", tmp_path / "libshim.so"
    src.write_text(SHIM % code)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(shim), str(src)], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, shim=str(shim))], capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, LD_PRELOAD=str(shim)))
    assert r.returncode == 0 and "same bits" in r.stdout, r.stderr[-2000:]
