"""Which batches take passes by themselves: large f32 ones whose instances have many
nodes to each node of their perimeters; small instances, the staged step (host logic,
no GPU)."""
import pytest


@pytest.fixture(scope="module")
def lbm():
    from paper_2005_08674_gb300 import build
    build.build()
    from paper_2005_08674_gb300 import lbm as m
    return m


@pytest.mark.parametrize("sizes,storage,bgk,mrt", [
    ([(8, 8)] * 20000, "f32", 0, 0), ([(64, 64)] * 300, "f32", 0, 0), ([(2000, 16)] * 40, "f32", 0, 0),
    ([(80, 80)] * 200, "f32", 0, 0), ([(100, 100)] * 120, "f32", 1, 0), ([(128, 128)] * 80, "f32", 1, 0),
    ([(160, 160)] * 50, "f32", 1, 1), ([(160, 160)] * 30, "f32", 0, 0),
    ([(1003, 900), (9, 8), (400, 301), (60, 257)], "f32", 1, 1), ([(1003, 900), (7, 8), (400, 301)], "f32", 0, 0),
    ([(160, 160)] * 50, "f16", 0, 0), ([(160, 160)] * 50, "f64", 0, 0)])
def test_picked_form(lbm, sizes, storage, bgk, mrt):
    b = lbm.lbm_batch_create([(nx, ny, 0.6, 1.0, 0.0, 0.0) for nx, ny in sizes], storage)
    try:
        assert lbm.lbm_batch_passes(b) == bgk
        lbm.lbm_batch_set_collision(b, "mrt", 1.4, 1.4, 1.2)
        assert lbm.lbm_batch_passes(b) == mrt
        lbm.lbm_batch_set_launch(b, 128, 3, 0, 1, 0, 128)
        assert lbm.lbm_batch_passes(b) == 0
    finally:
        lbm.lbm_batch_destroy(b)
