"""The FP64 forms' helpers against the plain operation that each stands for, bit for bit
(IEEE arithmetic of the host): the quotient by a kept reciprocal, the wrap into the box,
the conversions on the integer pipe, the lattice floor and the uniforms.  Random
significands, and the edges: zeros of both signs, infinities, NaN, subnormals, exponents
on both sides of every limit, all significand bits set, ties, 2^53, faces of the box."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "mpcd_internal.cuh"
using namespace mpcd;
__global__ void k_div(const double *a, const double *b, const double *rb, double *o, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) o[i] = div_by(a[i], b[i], rb[i]);
}
__global__ void k_one(int f, const double *x, const long long *v, double *o, int *w, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (f == 0) { w[i] = 0; o[i] = wrap_box(x[i], 12.0, w[i]); }
    if (f == 1) w[i] = __float_as_int(double_float(x[i]));
    if (f == 2) o[i] = i64_double(v[i]);
    if (f == 3) w[i] = lattice_floor(x[i]);
    if (f == 4) o[i] = u01d((uint32_t)v[i]);
    if (f == 5) o[i] = odd_of((uint32_t)v[i]);
}
extern "C" int run_div(const double *a, const double *b, const double *rb, double *o, int n)
{
    k_div<<<(n + 255) / 256, 256>>>(a, b, rb, o, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_one(int f, const double *x, const long long *v, double *o, int *w, int n)
{
    k_one<<<(n + 255) / 256, 256>>>(f, x, v, o, w, n);
    return (int)cudaDeviceSynchronize();
}
"""
RNG = np.random.default_rng(12)
N = 1 << 18
EDGES = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.2250738585072014e-308, 1.7976931348623157e308,
                  1.0, -1.0, 3.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52, 2.0 ** -400, 2.0 ** -401, 2.0 ** 399, 2.0 ** 400,
                  2.0 ** -1022, 2.0 ** 1023])


@pytest.fixture(scope="module")
def gpu(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import build_lib
    d = tmp_path_factory.mktemp("helpers")
    (d / "helpers.cu").write_text(SOURCE)
    subprocess.run([build_lib.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", *build_lib.ARCH,
                    "-I", build_lib.CSRC, "-I", os.path.join(build_lib.ROOT, "include"),
                    "-o", str(d / "helpers.so"), str(d / "helpers.cu")], check=True)
    lib = ctypes.CDLL(str(d / "helpers.so"))

    def up(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def ptr(t):
        return ctypes.c_void_p(t.data_ptr())

    def div(a, b, rb):
        t, o = [up(k) for k in (a, b, rb)], up(np.zeros(len(a)))
        assert lib.run_div(*[ptr(k) for k in t], ptr(o), len(a)) == 0
        return o.cpu().numpy()

    def one(f, x=None, v=None):
        n = len(x if x is not None else v)
        x, v = up(np.zeros(n) if x is None else x), up(np.zeros(n, np.int64) if v is None else v)
        o, w = up(np.zeros(n)), up(np.zeros(n, np.int32))
        assert lib.run_one(f, ptr(x), ptr(v), ptr(o), ptr(w), n) == 0
        return o.cpu().numpy(), w.cpu().numpy()

    return div, one


def values(lo, hi, n=N):
    return np.ldexp(RNG.uniform(1.0, 2.0, n), RNG.integers(lo, hi, n)) * RNG.choice([-1.0, 1.0], n)


def same(a, b, word=np.uint64):
    bits = (a.view(word) == b.view(word)) | (np.isnan(a) & np.isnan(b))
    assert bits.all(), (a[~bits][:4], b[~bits][:4])


@pytest.mark.parametrize("lo,hi", [(-4, 5), (-60, 61), (-420, 420), (-1080, 1024)])
def test_quotient(gpu, lo, hi):
    a, b = values(lo, hi), values(lo, hi)
    b[: N // 8] = np.ldexp(2.0 - 2.0 ** -52, RNG.integers(max(lo, -1000), min(hi, 1000), N // 8))
    ea, eb = np.meshgrid(EDGES, EDGES)
    a, b = np.concatenate([a, ea.ravel(), a[: 20]]), np.concatenate([b, eb.ravel(), EDGES])
    with np.errstate(all="ignore"):
        same(gpu[0](a, b, 1.0 / b), a / b)


def test_wrap(gpu):
    L = 12.0
    x = np.concatenate([RNG.uniform(-L, 2 * L, N), EDGES, [L, -L, 2 * L, np.nextafter(L, 0), np.nextafter(L, 99),
                        np.nextafter(-L, 0), np.nextafter(2 * L, 0), -1e-17, -1e-300, 3 * L, -2 * L]])
    with np.errstate(all="ignore"):
        y = np.where(x >= L, x - L, np.where(x < 0.0, np.where(x + L >= L, 0.0, x + L), x))
    got, bad = gpu[1](0, x=x)
    assert np.array_equal(bad != 0, ~((y >= 0.0) & (y < L)))
    same(got[bad == 0], y[bad == 0])


def test_to_float(gpu):
    ties = (np.float64(1.0) + np.arange(64) * 2.0 ** -24)[:, None] * 2.0 ** np.array([-126.0, -125.0, 0.0, 126.0])
    x = np.concatenate([values(-150, 130), EDGES, ties.ravel(), -ties.ravel(), np.nextafter(ties.ravel(), 0.0),
                        [2.0 ** 127, np.nextafter(2.0 ** 127, 0.0), np.nextafter(2.0 ** 128, 0.0),
                         np.nextafter(2.0 ** -126, 0.0)]])
    with np.errstate(all="ignore"):
        want = x.astype(np.float32)
    same(gpu[1](1, x=x)[1].view(np.float32), want, np.uint32)


def test_from_integers(gpu):
    v = RNG.integers(-2 ** 63, 2 ** 63 - 1, N) >> RNG.integers(0, 63, N)
    e = np.array([s * (2 ** k + d) for k in range(63) for d in (-1, 0, 1) for s in (-1, 1)] + [-2 ** 63, 2 ** 63 - 1],
                 dtype=np.int64)
    v = np.concatenate([v, e])
    same(gpu[1](2, v=v)[0], v.astype(np.float64))


def test_lattice_floor(gpu):
    k = RNG.integers(0, 2047 << 20, N)
    x = np.concatenate([RNG.uniform(0.0, 2047.0, N), k * 2.0 ** -20, np.nextafter(k * 2.0 ** -20, 4096.0),
                        np.maximum(0.0, np.nextafter(k * 2.0 ** -20, -1.0)), [0.0, -0.0, 5e-324, 2.0 ** -21]])
    assert np.array_equal(gpu[1](3, x=x)[1], np.floor(x * 2.0 ** 20).astype(np.int64))


def test_uniforms(gpu):
    v = np.concatenate([RNG.integers(0, 2 ** 32, N), [0, 1, 2, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 2, 2 ** 32 - 1]])
    same(gpu[1](4, v=v)[0], (v + 0.5) * 2.0 ** -32)
    same(gpu[1](5, v=v)[0], 2.0 * v + 1.0)
