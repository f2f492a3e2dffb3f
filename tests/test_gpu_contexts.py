"""Contexts beside one another and beside a caller's own CUDA work: threads, captured streams, work that
is still queued, device memory from a caller's allocator."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402


def test_contexts_step_in_two_threads():
    """Tiles of two heights at once, in launches of 2, 3 and 4 steps: what each alone gives."""
    sizes, calls, got, errors = ((500, 500), (128, 128)), 3000, {}, []

    def work(size):
        try:
            stream = torch.cuda.Stream()
            with Cavity(*size, Re=300.0, U=0.1, dtype="f32s", stream=stream) as cav:
                for k in range(calls):
                    cav.step(2 + k % 3)
                got[size] = cav.populations(host=True)
        except Exception as e:
            errors.append(f"{size}: {e}")

    threads = [threading.Thread(target=work, args=(s,)) for s in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for size in sizes:
        with Cavity(*size, Re=300.0, U=0.1, dtype="f32s") as cav:
            cav.step(3 * calls)
            assert (cav.populations(host=True) == got[size]).all(), size


@pytest.mark.parametrize("calls", [(2,), (4,), (12,), (3, 5), (20, 40), (1, 7, 6)])
@pytest.mark.parametrize("dtype,cfg", [("f32s", 7), ("f32s", 6), ("f16s", 7), ("f64", 5)])
def test_replays_of_captured_steps_advance(dtype, cfg, calls):
    """Calls of an even number of steps together, captured once by the caller and replayed."""
    stream, replays = torch.cuda.Stream(), 5
    with Cavity(150, 70, Re=300.0, U=0.1, dtype=dtype, stream=stream) as cav, \
            Cavity(150, 70, Re=300.0, U=0.1, dtype=dtype) as ref:
        B.lbm_set_launch_config(cav.ctx, cfg)
        cav.step(7)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for n in calls:
                cav.step(n)
        torch.cuda.synchronize()
        for _ in range(replays):
            graph.replay()
        torch.cuda.synchronize()
        for _ in range(7 + sum(calls) * replays):
            ref.step(1)
        assert np.array_equal(cav.populations(host=True), ref.populations(host=True))


@pytest.mark.parametrize("cfg", [5, 6, 7])
def test_steps_beside_a_capture_of_another_stream(cfg):
    """Calls that capture a part or an interval of their own, launched directly and replayed, while the
    caller captures something else: both go on."""
    x = torch.zeros(1000, device="cuda")
    with Cavity(150, 70, Re=300.0, U=0.1, dtype="f32s", stream=torch.cuda.Stream()) as cav, \
            Cavity(150, 70, Re=300.0, U=0.1, dtype="f32s") as ref:
        start = ref.moments()
        B.lbm_set_launch_config(cav.ctx, cfg)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
            x += 1
            for _ in range(3):
                cav.set_moments(*start)
                cav.step(7)
            cav.step(93)
            cav.step(100)
            x += 1
        graph.replay()
        ref.set_moments(*start)
        ref.step(200)
        torch.cuda.synchronize()
        assert float(x.sum()) == 2000.0
        assert np.array_equal(cav.populations(host=True), ref.populations(host=True))


def test_steps_do_not_wait_for_queued_work():
    """More parts than are kept, each captured, then others behind half a second of queued work: the
    calls return before that work ends, and the state is what one call gives."""
    stream = torch.cuda.Stream()
    with Cavity(150, 70, Re=300.0, U=0.1, dtype="f32s", stream=stream) as cav, \
            Cavity(150, 70, Re=300.0, U=0.1, dtype="f32s") as ref:
        start = ref.moments()
        torch.cuda.synchronize()
        for n in range(4, 24):
            for _ in range(2):
                cav.set_moments(*start)
                cav.step(n)
        stream.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(1_000_000_000)
            slept = stream.record_event()
            for n in range(24, 30):
                for _ in range(2):
                    cav.set_moments(*start)
                    cav.step(n)
            assert not slept.query()
        for n in range(30, 80):
            for _ in range(3):
                cav.set_moments(*start)
                cav.step(n)
        ref.set_moments(*start)
        ref.step(79)
        assert np.array_equal(cav.populations(host=True), ref.populations(host=True))
