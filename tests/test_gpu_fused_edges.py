"""Edges of the fused shapes: the shift of the taller tiles in both directions, probes on every wall and
corner, the last strip and the last tile one column or row wide."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402


def run(nx, ny, dtype, cfg, points):
    with Cavity(nx, ny, tau=0.58, U=0.1, dtype=dtype, corners_moving=True) as cav:
        B.lbm_set_launch_config(cav.ctx, cfg)
        series = [cav.probe(x, y, every=e, cap=120)[1] for x, y, e in points]
        for n in (10, 3, 90, 17):
            cav.step(n)
        return cav.populations(host=True), [s.cpu().numpy() for s in series]


@pytest.mark.parametrize("nx,ny", [(500, 241), (505, 265), (481, 409)])  # over 304 low tiles: 24 rows a tile
@pytest.mark.parametrize("dtype", ["f32", "f32s", "bf16s", "q16s"])
def test_taller_tiles_and_probes_on_the_walls(nx, ny, dtype):
    top, right = (ny - 1) / nx, (nx - 1) / nx
    for points in (((0.0, 0.3 * top, 1), (right, 0.5 * top, 2), (0.5, top, 1), (0.5, 0.0, 3)),
                   ((0.0, 0.0, 1), (right, 0.0, 1), (0.0, top, 1), (right, top, 1))):
        want, probes = run(nx, ny, dtype, 0, points)
        for cfg in (6, 7):
            got, p = run(nx, ny, dtype, cfg, points)
            assert np.array_equal(got, want), cfg
            for a, b in zip(p, probes):
                assert np.array_equal(a, b), cfg
