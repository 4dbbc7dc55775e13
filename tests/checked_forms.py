"""Driver for the bounds-checked library (run in a child process with LBM_CHECKED=1 by
test_forms_gpu.py; not collected by pytest): the launch forms of several steps --
tiles, resident domains, the form lbm_step picks, batched passes -- on small, ragged
and periodic domains.  Prints one JSON line: whether the library is the checked build,
how many accesses it rejected and the first rejected address."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import torch  # noqa: E402

from paper_2005_08674_gb300 import inputs, lbm  # noqa: E402

SIZES = [(8, 8), (9, 13), (17, 200), (131, 75), (257, 9), (130, 66)]
KWS = [dict(beta=0.1), dict(farfield_u=(0.02, 0.01), corner_mode=1, grad_order=2, collision="mrt"),
       dict(edges=[("velocity", 0.03, 0.0), "nsbc", "periodic", "periodic"]), dict(edges=["periodic"] * 4)]


def main():
    torch.cuda.set_device(0)
    for nx, ny in SIZES:
        fields = inputs.acoustic_pulse(nx, ny, 1e-3, 2.0, [((nx - 1) / 2, (ny - 1) / 2)])
        for storage in ("f64", "f32", "f16", "bf16"):
            for kw in KWS:
                for tiles in (True, False):
                    with lbm.Simulation(nx, ny, 0.6, storage=storage, **kw) as s:
                        s.init(*fields)
                        if tiles:
                            s.set_tiles()
                        s.step(70).step(21).status()
                        s.macros()
    ws = inputs.batch_instances(count=6, lo=8, hi=90)
    for storage in ("f32", "f16"):
        for corner in (0, 1):
            with lbm.Batch(ws, storage=storage, beta=0.05, corner_mode=corner) as b:
                for k, w in enumerate(ws):
                    b.init(k, *w.fields())
                b.set_twostep(True)
                for n in (21, 2, 3, 5):
                    b.step(n)
                b.status()
                for k in range(len(ws)):
                    b.macros(k)
    torch.cuda.synchronize()
    checked, rejected, first = lbm.lbm_check_read()
    print(json.dumps(dict(checked=checked, rejected=rejected, first=hex(first))), flush=True)


if __name__ == "__main__":
    main()
