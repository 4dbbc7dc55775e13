"""A scratch area is the caller's between two calls: handles of different size may
share one, the caller may write to it, and steps on two streams do not meet in it.
Each run must give the bits of a handle that has an area of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


class Handle:
    """A domain on its own buffers and the given scratch area."""

    def __init__(self, lbm, nx, ny, storage, scratch, fields, stream):
        import torch
        self.lbm, self.h = lbm, lbm.lbm_create(nx, ny, 0.6)
        lbm.lbm_set_precision(self.h, storage)
        lbm.lbm_set_stream(self.h, stream.cuda_stream)
        self.bufs = [torch.empty(lbm.lbm_buffer_bytes(self.h), dtype=torch.uint8, device="cuda") for _ in range(2)]
        assert scratch.numel() >= lbm.lbm_scratch_bytes(self.h)
        lbm.lbm_bind(self.h, self.bufs[0].data_ptr(), self.bufs[1].data_ptr(), scratch.data_ptr())
        self.fields = [torch.tensor(a, device="cuda") for a in fields]
        torch.cuda.synchronize()
        lbm.lbm_init_device(self.h, *[t.data_ptr() for t in self.fields])
        self.shape = (ny, nx)

    def step(self, n):
        self.lbm.lbm_step(self.h, n)

    def macros(self):
        out = [np.empty(self.shape) for _ in range(3)]
        self.lbm.lbm_get_macros(self.h, *out)
        return out

    def close(self):
        self.lbm.lbm_destroy(self.h)


def _fields(nx, ny):
    rng = np.random.default_rng(nx)
    return [b + 1e-3 * rng.standard_normal((ny, nx)) for b in (1.0, 0.0, 0.0)]


def _alone(lbm, nx, ny, storage, steps):
    with lbm.Simulation(nx, ny, 0.6, storage=storage) as s:
        s.init(*_fields(nx, ny)).set_launch(128, 1, 0)
        return s.step(steps).macros()


# a pass and a resident domain, next to one a little larger
@pytest.mark.parametrize("nx,ny,storage", [(1201, 1003, "f32"), (1801, 1600, "f16"), (300, 300, "f32")])
@pytest.mark.parametrize("way", ["handles", "caller", "streams"])
def test_shared_scratch(lbm, nx, ny, storage, way):
    import torch
    big = (nx + 60, ny + 60)
    need = lbm.lbm_create(*big, 0.6)
    scratch = torch.empty(lbm.lbm_scratch_bytes(need), dtype=torch.uint8, device="cuda")
    lbm.lbm_destroy(need)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    a = Handle(lbm, nx, ny, storage, scratch, _fields(nx, ny), streams[0])
    b = Handle(lbm, *big, storage, scratch, _fields(*big), streams[0 if way == "handles" else 1])
    torch.cuda.synchronize()
    for _ in range(3):
        a.step(70)
        if way == "handles":
            b.macros()  # fills the area with b's fields
        elif way == "streams":
            b.step(70)
        else:
            torch.cuda.synchronize()
            scratch.fill_(0x5A)
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    for x, y in zip(a.macros(), _alone(lbm, nx, ny, storage, 210)):
        assert np.array_equal(x, y)
    if way == "streams":
        for x, y in zip(b.macros(), _alone(lbm, *big, storage, 210)):
            assert np.array_equal(x, y)
    a.close()
    b.close()
