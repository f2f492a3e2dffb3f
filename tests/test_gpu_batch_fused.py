"""When a batch fuses its plain steps, and that what it gives then is what single cavities give."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402


def rows_that_fuse():
    """Twice the strip-rows from which plain steps are fused: 8 a warp, 4 warps a block, 3 blocks an SM."""
    return 2 * 8 * 4 * 3 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("nx,f32,f32s", [(500, 3, 3), (240, 3, 3), (150, 3, 3), (64, 3, 3),  # as many strips as the row step's, or 5 to its 4
                                         (121, 1, 3), (128, 1, 3)])                         # two strips to one
def test_fusing_follows_the_strips(nx, f32, f32s):
    n = 40
    ny = -(-rows_that_fuse() // n)
    for dtype, want in (("f32", f32), ("f32s", f32s), ("f64", 1), ("f16s", 1)):
        b = B.lbm_batch_create([nx] * n, [ny] * n, [2.0 * nx] * n, [0.1] * n, dtype)
        try:
            assert B.lbm_batch_steps_per_pass(b) == want, dtype
        finally:
            B.lbm_batch_destroy(b)
    b = B.lbm_batch_create([nx], [40], [2.0 * nx], [0.1], "f32s")
    try:
        assert B.lbm_batch_steps_per_pass(b) == 1
    finally:
        B.lbm_batch_destroy(b)


@pytest.mark.parametrize("dtype", ["f32", "f32s"])
def test_batch_that_is_known_to_fuse_equals_single_cavities(dtype):
    """Graph replays, leftover steps and retirement, fused from first to last step (no tuning, whose timing
    could choose otherwise)."""
    n = 16
    cases = [(130, -(-rows_that_fuse() // (2 * n)) + i, 300.0 + 50 * i, 0.1) for i in range(n)]
    cases += [(3, 5, 10.0, 0.1), (121, 40, 200.0, 0.1), (241, 73, 500.0, 0.1)]
    nx, ny, re, u = zip(*cases)
    b = B.lbm_batch_create(nx, ny, re, u, dtype)
    B.lbm_batch_set_stream(b, torch.cuda.current_stream().cuda_stream)
    try:
        for steps in (100, 37, 114):
            assert B.lbm_batch_steps_per_pass(b) == 3
            B.lbm_batch_step(b, steps)
        assert B.lbm_batch_steps_per_pass(b) == 3
        for i, (x, y, e, v) in enumerate(cases):
            with Cavity(x, y, Re=e, U=v, dtype=dtype) as cav:
                B.lbm_set_launch_config(cav.ctx, 0)
                cav.step(251)
                got = torch.empty((9, y, x), dtype=torch.float64, device="cuda")
                B.lbm_batch_get_populations(b, i, got)
                assert torch.equal(got, cav.populations()), i
        rc, done = B.lbm_batch_run_to_residual(b, len(cases), 10.0, 200)  # everything retires at the next checkpoint
        assert rc == B.LBM_OK and (done == 49).all()
        assert B.lbm_batch_steps_per_pass(b) == 1
    finally:
        B.lbm_batch_destroy(b)
