"""The FP64 form's Gamma(n_dof / 2) draw against the host's extended precision, cell by cell
from the same Philox words: a sum of exponentials and, for an odd number of degrees
of freedom, half a squared normal.  The largest relative error over 2e5 cells must stay
below that of a correctly rounded logarithm for each uniform and their plain sum, which
is (k + 1) 2^-53 for k terms; with few uniforms the sum can be small, and rounding errors in a
product of them would show there."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "kernels_solvent.cu"
namespace mpcd {
__global__ void k_gamma(double *o, uint32_t *words, int n_dof, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    DevReplica r{};
    r.key0 = 12345u;
    r.key1 = 678u;
    o[i] = gamma_half_dof(r, 7, (uint32_t)i, n_dof, 0.0);
    for (int e = 0; e < n_dof / 2; ++e) {
        const uint4 w = draw(r, 7, (uint32_t)i, TAG_THERMO, (uint32_t)(e >> 2));
        words[(size_t)e * n + i] = e % 4 == 0 ? w.x : e % 4 == 1 ? w.y : e % 4 == 2 ? w.z : w.w;
    }
}
}
extern "C" int run_gamma(double *o, uint32_t *words, int n_dof, int n)
{
    mpcd::k_gamma<<<(n + 255) / 256, 256>>>(o, words, n_dof, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def gamma(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import build_lib
    d = tmp_path_factory.mktemp("gamma")
    (d / "gamma.cu").write_text(SOURCE)
    subprocess.run([build_lib.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", *build_lib.ARCH,
                    "-I", build_lib.CSRC, "-I", os.path.join(build_lib.ROOT, "include"),
                    "-o", str(d / "gamma.so"), str(d / "gamma.cu")], check=True)
    lib = ctypes.CDLL(str(d / "gamma.so"))

    def run(n_dof, n):
        o = torch.zeros(n, dtype=torch.float64, device="cuda")
        w = torch.zeros(max(1, n_dof // 2), n, dtype=torch.int32, device="cuda")
        assert lib.run_gamma(ctypes.c_void_p(o.data_ptr()), ctypes.c_void_p(w.data_ptr()), n_dof, n) == 0
        return o.cpu().numpy(), w.cpu().numpy().view(np.uint32)
    return run


@pytest.mark.parametrize("n_dof", [6, 8, 12, 18, 24, 30, 36, 66])
def test_error_of_the_sum(gamma, n_dof):
    if np.finfo(np.longdouble).eps > 2.0 ** -62:
        pytest.skip("no extended precision on this host")
    g, words = gamma(n_dof, 200000)
    u = (words.astype(np.longdouble) + np.longdouble(0.5)) * np.longdouble(2.0) ** -32
    want = -np.log(u).sum(axis=0)
    assert (np.abs(g - want) / want).astype(float).max() <= (n_dof // 2 + 1) * 2.0 ** -53
