"""Device memory that a caller's allocator aligns to 8 bytes and no more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402
from paper_2211_05009_gb300.cavity import Cavity  # noqa: E402


class OffsetAllocator:
    """Buffers that begin 8 bytes past a 256-byte boundary."""

    def __init__(self):
        self.live = {}
        self.alloc_fn, self.release_fn = B.ALLOC_FN(self._alloc), B.RELEASE_FN(self._release)

    def _alloc(self, nbytes, user):
        buf = torch.zeros(int(nbytes) + 256, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        assert buf.data_ptr() % 256 == 0
        self.live[buf.data_ptr() + 8] = buf
        return buf.data_ptr() + 8

    def _release(self, ptr, user):
        del self.live[ptr]


@pytest.mark.parametrize("nx,ny", [(133, 77), (1300, 1100)])  # tiles and the march by default in LBM_F32S
@pytest.mark.parametrize("dtype", ["f32", "f32s", "f64"])
def test_memory_aligned_to_8_bytes(nx, ny, dtype):
    def run(cav):
        out = []
        for cfg in (None, 6, 7, "tuned"):
            if cfg == "tuned":
                B.lbm_autotune(cav.ctx, 4)
            elif cfg is not None:
                B.lbm_set_launch_config(cav.ctx, cfg)
            cav.step(39)
            out.append(cav.populations(host=True))
        return out

    with Cavity(nx, ny, Re=500.0, U=0.1, dtype=dtype) as cav:
        want = run(cav)
    a = OffsetAllocator()
    B.lbm_set_allocator(a.alloc_fn, a.release_fn)
    try:
        with Cavity(nx, ny, Re=500.0, U=0.1, dtype=dtype) as cav:
            assert a.live
            got = run(cav)
    finally:
        B.lbm_set_allocator(None, None)
    assert not a.live
    for x, y in zip(got, want):
        assert np.array_equal(x, y)
