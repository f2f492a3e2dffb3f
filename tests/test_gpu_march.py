"""Launch shapes that advance several steps per launch against the single-step shape: populations
and probe samples bitwise, Eq. 6 to the rounding of its differently grouped FP32 partial sums, at
the sizes where strips, halos and segments can go wrong."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402

SIZES = [(3, 3), (5, 4), (66, 9), (121, 40),   # one strip; two-row segments; the wall one past a strip
         (129, 31), (130, 33), (131, 34), (240, 65),  # right wall in every slot of a lane; exactly two strips
         (500, 200)]


def run(nx, ny, dtype, cfg, corners):
    with Cavity(nx, ny, tau=0.62, U=0.1, dtype=dtype, corners_moving=corners) as cav:
        B.lbm_set_launch_config(cav.ctx, cfg)
        top = (ny - 1) / nx  # probes on the lid, on the bottom wall and inside, sampled at odd steps too
        series = [cav.probe(x, y, every=e, cap=250)[1] for x, y, e in ((0.5, top, 3), (0.4, 0.0, 2), (0.3, 0.4 * top, 1))]
        for n in (37, 2, 1, 160, 50):  # crosses two checkpoints off and on the interval boundary
            cav.step(n)
        assert cav.step_count == 250
        return cav.populations(host=True), [s.cpu().numpy() for s in series], cav.residual()


@pytest.mark.parametrize("dtype", ["f32", "f32s", "f16s", "bf16s", "f64", "q16s"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_fused_steps_equal_single_steps(nx, ny, dtype):
    want, probes, r = run(nx, ny, dtype, 0, corners=nx == 129)
    assert np.isfinite(want).all()
    for cfg in range(1, B.lbm_launch_config_count()):
        got, p, rc = run(nx, ny, dtype, cfg, corners=nx == 129)
        assert np.array_equal(got, want), f"shape {cfg}"
        for a, b in zip(p, probes):
            assert np.array_equal(a, b), f"shape {cfg}"
        assert abs(rc - r) <= (1e-12 if dtype == "f64" else 2e-6) * r, f"shape {cfg}"


def test_state_moves_between_shapes():
    """A shape changed between calls, a re-seed and a checkpoint file continue from the current state."""
    out = []
    for shapes in ((0, 0, 0), (6, 6, 0), (1, 6, 6)):
        with Cavity(150, 70, Re=300.0, U=0.1, dtype="f32s") as cav:
            for cfg, n in zip(shapes, (153, 100, 47)):
                B.lbm_set_launch_config(cav.ctx, cfg)
                cav.step(n)
            fields = cav.moments()
            first = cav.populations(host=True)
            cav.set_moments(*fields)
            cav.step(200)
            out.append((first, cav.populations(host=True), cav.residual()))
    for first, second, r in out[1:]:
        assert np.array_equal(first, out[0][0]) and np.array_equal(second, out[0][1])
        assert abs(r - out[0][2]) <= 2e-6 * r


@pytest.mark.parametrize("dtype", ["f32", "f32s"])
def test_fused_batch_equals_single_cavities(dtype):
    """A batch with rows enough to fuse its plain steps (uneven cavities, the smallest grid and one
    whose right wall is alone in its strip among them), with probes, over graph replays, leftover
    steps, a tile-shape trial in between and retirement."""
    cases = [(130, 900 + 17 * i, 300.0 + 50 * i, 0.1) for i in range(8)] + [(3, 5, 10.0, 0.1), (121, 40, 200.0, 0.1), (241, 333, 500.0, 0.1)]
    every, cap, n = 3, 200, len(cases)
    nx, ny, re, u = zip(*cases)
    b = B.lbm_batch_create(nx, ny, re, u, dtype)
    B.lbm_batch_set_stream(b, torch.cuda.current_stream().cuda_stream)
    series = torch.zeros((n, cap, 2), dtype=torch.float64, device="cuda")
    try:
        B.lbm_batch_probe(b, [0.5] * n, [0.3] * n, every, series, cap)
        B.lbm_batch_step(b, 100)
        B.lbm_batch_step(b, 37)
        B.lbm_batch_autotune(b, 7)
        B.lbm_batch_step(b, 214)
        r, status = B.lbm_batch_residual(b, n)
        assert (status == 0).all()
        for i, (x, y, e, v) in enumerate(cases):
            with Cavity(x, y, Re=e, U=v, dtype=dtype) as cav:
                B.lbm_set_launch_config(cav.ctx, 0)
                ser = cav.probe(0.5, 0.3, every=every, cap=cap)[1]
                cav.step(351)
                got = torch.empty((9, y, x), dtype=torch.float64, device="cuda")
                B.lbm_batch_get_populations(b, i, got)
                assert torch.equal(got, cav.populations()), f"cavity {i}"
                assert torch.equal(series[i, :351 // every], ser[:351 // every]), f"cavity {i}"
                assert abs(r[i] - cav.residual()) <= 2e-6 * r[i]
        rc, done = B.lbm_batch_run_to_residual(b, n, 10.0, 200)  # everything retires at the next checkpoint
        assert rc == B.LBM_OK and (done == 49).all()
    finally:
        B.lbm_batch_destroy(b)


@pytest.mark.parametrize("dtype,cfg", [("f32s", 6), ("f32s", 2), ("f64", 5)])
def test_repeated_parts_equal_one_call(dtype, cfg):
    """The same few steps again and again (captured at their second sight, across checkpoints and past
    the number of parts that are kept) give what one call of all of them gives."""
    with Cavity(150, 70, Re=300.0, U=0.1, dtype=dtype) as a, Cavity(150, 70, Re=300.0, U=0.1, dtype=dtype) as b:
        for c in (a, b):
            B.lbm_set_launch_config(c.ctx, cfg)
        sa, sb = (c.probe(0.5, 0.3, every=3, cap=700)[1] for c in (a, b))
        total = 0
        for k in range(40):
            for n in (7, 20, 3 + k % 5):
                a.step(n)
                total += n
        b.step(total)
        assert a.step_count == b.step_count == total
        assert torch.equal(a.populations(), b.populations()) and torch.equal(sa, sb)
        assert a.residual() == b.residual()


@pytest.mark.parametrize("nx", [3, 31, 32, 33, 63, 64, 65, 96, 97])
def test_f64_ragged_widths_match_oracle(nx):
    """One node per lane: widths around multiples of a strip, single and batched, against the oracle.

    120 steps; the oracle rounds each operation to 2^-53, this code too, so populations agree to about
    120 x 10 roundings of 1.1e-16: 1e-12 holds eight times that."""
    ny, steps = 21, 120
    p = O.Params(nx, ny, 3 * 0.1 * nx / 60.0 + 0.5, 0.1)
    want = O.to_soa(O.run(p, O.init(p), steps))
    with Cavity(nx, ny, tau=p.tau, U=0.1, dtype="f64") as cav:
        cav.step(steps)
        got = cav.populations(host=True)
        fields = [f.clone() for f in cav.moments()]
    assert (np.abs(got - want) / np.abs(want)).max() < 1e-12
    b = B.lbm_batch_create([nx, 40], [ny, 9], [60.0, 50.0], [0.1, 0.1], "f64")
    try:
        B.lbm_batch_step(b, steps)
        out = [torch.empty_like(f) for f in fields]
        B.lbm_batch_moments(b, 0, *out)
    finally:
        B.lbm_batch_destroy(b)
    for a, f in zip(out, fields):
        assert torch.equal(a, f)
