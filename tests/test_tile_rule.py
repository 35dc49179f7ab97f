"""The FP64 form's tile rule: the shapes of grids from the smallest to the
largest, for every instance, and the grids that other tests take for a shape."""
import shutil

import pytest

from .tile_rule import shape

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")


@pytest.mark.parametrize("cons,viscous", [(False, False), (False, True), (True, False), (True, True)])
def test_shapes_from_small_to_large(cons, viscous):
    kw = {"cons": cons, "viscous": viscous}
    for n in (6, 16, 37, 64):
        assert shape(n, n, **kw) == "8x4"
    assert shape(123, 101, **kw) == "16x8"  # one wave of 104 tiles
    for n in (1024, 4096, 46340):
        assert shape(n, n, **kw) in ("16x15", "16x8")
    assert shape(1024, 1024, **kw) == "16x15"
    for nx, ny in ((6, 1 << 28), (1 << 28, 6), (12, 990000), (8, 300000)):  # no overflow, some shape
        assert shape(nx, ny, **kw) in ("16x15", "16x8", "8x4")


def test_the_instances_differ():
    # 80^2: 50 tiles of 16 x 8 beat 200 of 8 x 4 only where one CTA fills an SM
    assert shape(80, 80) == "8x4" and shape(80, 80, cons=True, viscous=True) == "16x8"
    # one tile of 16 x 8 more than SMs
    assert shape(136, 136) == "8x4" and shape(136, 136, viscous=True) == "16x8"


def test_a_size_that_names_a_shape_it_does_not_take():
    # (tests/test_gpu_tiles.py lists 190 x 117 for 16 x 8)
    assert shape(190, 117) == "16x15"
