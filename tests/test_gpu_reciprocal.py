"""The FP64 step's reciprocal against CUDA's correctly rounded one: the library's header compiled into a
kernel of its own."""
import ctypes
import importlib
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

build = importlib.import_module("paper_2211_05009_gb300.build")

SOURCE = r"""
#include "lbm_step_kernel.cuh"
__global__ void k(const double* v, double* ours, double* exact, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    ours[i] = -lbm::nrcp(v[i], 1.0);
    exact[i] = __drcp_rn(v[i]);
}
extern "C" int reciprocals(const double* v, double* ours, double* exact, int n) {
    k<<<(n + 255) / 256, 256>>>(v, ours, exact, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    d = tmp_path_factory.mktemp("reciprocal")
    src, lib = os.path.join(d, "r.cu"), os.path.join(d, "r.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-shared", "-o", lib, src], check=True, capture_output=True)
    fn = ctypes.CDLL(lib).reciprocals

    def call(v):
        v = torch.tensor(v, dtype=torch.float64, device="cuda")
        out = torch.empty((2, v.numel()), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(ctypes.c_void_p(v.data_ptr()), ctypes.c_void_p(out[0].data_ptr()), ctypes.c_void_p(out[1].data_ptr()), v.numel()) == 0
        return out.cpu().numpy()

    return call


def test_reciprocal_is_the_nearest_or_beside_it(reciprocals):
    """An estimate within 2^-19 leaves e^3 <= 2^-57 beside the one rounding of the last operation, an eighth of
    half a unit: never more than one unit from the nearest."""
    r = np.random.RandomState(5)
    bits = (r.randint(0, 1 << 52, 400000, dtype=np.int64) | (r.randint(1023 - 1000, 1023 + 1000, 400000) << 52))
    v = np.concatenate([r.uniform(0.5, 2.0, 400000), 1.0 + r.uniform(-0.05, 0.05, 400000), bits.view(np.float64),
                        np.nextafter(2.0 ** np.arange(-60, 60), 0), 2.0 ** np.arange(-60, 60)])
    v = np.concatenate([v, -v])
    ours, exact = reciprocals(v)
    assert np.abs(ours.view(np.int64) - exact.view(np.int64)).max() <= 1


def test_reciprocal_of_what_is_no_number(reciprocals):
    ours, _ = reciprocals([np.inf, -np.inf, np.nan, 0.0])
    assert not np.isfinite(ours).any()
