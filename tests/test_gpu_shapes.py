"""The launch shape of a new context on grids whose width the march's strips fill badly."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402

MARCH, TILE = 6, 7


@pytest.mark.parametrize("nx,ny,f32,f32s", [
    (2048, 2048, MARCH, MARCH), (361, 5000, MARCH, MARCH),                     # strips filled
    (160, 12000, TILE, TILE), (121, 20000, TILE, TILE), (20, 60000, TILE, TILE),  # two strips for little more than one; one for 20
    (1000, 1000, 5, MARCH), (121, 10000, 5, TILE), (500, 1000, 2, TILE)])      # f32: row shapes within the L2 cache
def test_default_shape(nx, ny, f32, f32s):
    for dtype, want in (("f32", f32), ("f32s", f32s)):
        with Cavity(nx, ny, tau=0.6, U=0.1, dtype=dtype) as cav:
            assert cav.info.launch_config == want, dtype
