"""lbm_step and lbm_batch_step in a graph that the caller captures: replays of an even
number of steps go on from one another, whatever form the steps are launched in."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


def _fields(nx, ny, seed=1):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.zeros((3, ny, nx), dtype=torch.float64, device="cuda")
    f[0] = 1.0 + 1e-3 * torch.rand((ny, nx), dtype=torch.float64, device="cuda", generator=g)
    return f


def _replay(step, n, stream, times=3):
    import torch
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        step(n)
    for _ in range(times):
        g.replay()
    torch.cuda.synchronize()


# tiles, one launch per step (resident from 64 steps on), f64, passes in both widths
@pytest.mark.parametrize("nx,ny,storage", [(64, 40, "f32"), (300, 300, "f32"), (500, 500, "f16"), (200, 200, "f64"),
                                           (1201, 1003, "f32"), (1801, 1600, "f16")])
@pytest.mark.parametrize("n", [2, 4, 6, 12, 14, 16, 70])
def test_replayed_domain(lbm, nx, ny, storage, n):
    import torch
    f = _fields(nx, ny)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with lbm.Simulation(nx, ny, 0.6, storage=storage, stream=stream) as s:
        s.init_device(f[0], f[1], f[2]).step(n)
        s.init_device(f[0], f[1], f[2])
        _replay(s.step, n, stream)
        got = s.populations()
    with lbm.Simulation(nx, ny, 0.6, storage=storage) as s:
        ref = s.init_device(f[0], f[1], f[2]).set_launch(128, 1, 0).step(3 * n).populations()
    assert (got == ref).all()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n", [2, 4, 6, 16])
def test_replayed_batch(lbm, storage, n):
    import torch

    class W:
        farfield_rho, farfield_u, tau = 1.0, (0.0, 0.0), 0.6

        def __init__(self, nx, ny):
            self.nx, self.ny = nx, ny
    ws = [W(1003, 1001), W(400, 301)]
    fields = [_fields(w.nx, w.ny).cpu().numpy() for w in ws]
    stream = torch.cuda.Stream()
    out = []
    for replay in (True, False):
        with lbm.Batch(ws, storage=storage, stream=stream) as b:
            if replay:
                for k, f in enumerate(fields):
                    b.init(k, *f)
                b.step(n)
                torch.cuda.synchronize()
            for k, f in enumerate(fields):
                b.init(k, *f)
            if replay:
                _replay(b.step, n, stream)
            else:
                b.step(3 * n)
            b.status()
            out.append([b.macros(k) for k in range(len(ws))])
    for x, y in zip(*out):
        assert all((p == q).all() for p, q in zip(x, y))
