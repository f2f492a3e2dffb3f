"""The network's buffers and captured passes over a history of sample sizes and back ends."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2211_05009_gb300 import binding as B  # noqa: E402


def make(width=4, backend=3):
    n = B.lbm_net_create(width, 3)
    B.lbm_net_set_backend(n, backend)
    B.lbm_net_set_stream(n, torch.cuda.current_stream().cuda_stream)
    return n


def sample(H, W):
    g = torch.Generator(device="cuda").manual_seed(H * 1000 + W)
    return torch.rand((7, H, W), generator=g, device="cuda") - 0.5


def forward(n, H, W):
    out = torch.empty((3, H, W), dtype=torch.float32, device="cuda")
    B.lbm_net_forward(n, sample(H, W), H, W, out)
    return out


def test_results_do_not_depend_on_the_sizes_before():
    """Growing and shrinking buffers, more sizes than graphs are kept for, the same size again under other
    back ends: always what a network that saw nothing else gives."""
    small = [(16 * k, 128) for k in range(1, 21)]
    history = [(64, 128)] * 3 + [(512, 512)] * 3 + [(16, 128)] * 3 + [(256, 384)] * 2 + small * 2 + [(64, 128)] * 3
    want = {}
    for size in set(history):
        n = make()
        want[size] = forward(n, *size)
        B.lbm_net_destroy(n)
    n, other = make(), {}
    for size in history:
        assert torch.equal(forward(n, *size), want[size]), size
    for backend in (1, 3, 1, 3):
        B.lbm_net_set_backend(n, backend)
        for _ in range(2):
            got = forward(n, 64, 128)
            assert torch.equal(got, other.setdefault(backend, got)), backend
    assert torch.equal(other[3], want[64, 128])
    B.lbm_net_destroy(n)


def test_memory_of_a_large_sample_is_given_back():
    n = make(width=8)
    try:
        forward(n, 16, 128)
        inputs = sample(1024, 1024), torch.empty((3, 1024, 1024), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        B.lbm_net_forward(n, inputs[0], 1024, 1024, inputs[1])
        torch.cuda.synchronize()
        large = torch.cuda.mem_get_info()[0]
        forward(n, 16, 128)
        torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        assert before - large > 200 << 20  # the sample's tensors alone: 1024^2 pixels, 8 channels and more, 4 bytes, twice
        assert after - large > 0.9 * (before - large)
    finally:
        B.lbm_net_destroy(n)
