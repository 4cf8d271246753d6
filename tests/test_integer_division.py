"""div_by and sqrt_int (csrc/ddiv.cuh) against the IEEE operations.

On the host, with approximations one unit in the last place below, at and
above the exact value (the integer steps have to put right what the FP32
unit's documented error allows); on the GPU, with the unit's own, over every
input that they can get."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_05975_gb300", "csrc")

HOST = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>
template <typename A, typename B> static A bits(B b) { A a; static_assert(sizeof a == sizeof b, ""); memcpy(&a, &b, sizeof a); return a; }
static int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)bits<uint64_t>(x); }
static unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
static int __mulhi(int a, int b) { return (int)(((int64_t)a * b) >> 32); }
static float __uint_as_float(unsigned x) { return bits<float>(x); }
static unsigned __float_as_uint(float x) { return bits<unsigned>(x); }
static double __longlong_as_double(long long x) { return bits<double>(x); }
static int g_ulp;
namespace lu {
static float approx_rcp(float x) { return bits<float>(bits<unsigned>((float)(1.0 / x)) + g_ulp); }
static float approx_rsqrt(float x) { return bits<float>(bits<unsigned>((float)(1.0 / std::sqrt((double)x))) + g_ulp); }
static double hardware_div(double a, double b) { return a / b; }
static double hardware_sqrt(double x) { return std::sqrt(x); }
}
#include "ddiv.cuh"
extern "C" long long check(int op, int ulp, long long n, const double* a, const double* b, double* where) {
    g_ulp = ulp;
    long long bad = 0;
    for (long long i = 0; i < n; ++i) {
        const double want = op ? std::sqrt(a[i]) : a[i] / b[i];
        const double got = op ? lu::sqrt_int(a[i]) : lu::div_by(a[i], b[i], lu::div_rec(b[i]));
        if (bits<uint64_t>(want) != bits<uint64_t>(got) && !(want != want && got != got)) {
            if (!bad) { where[0] = a[i]; where[1] = b[i]; where[2] = got; }
            ++bad;
        }
    }
    return bad;
}
"""

GPU = r"""
#include <cuda_runtime.h>
#include "ddiv.cuh"
// every leading 24 bits of a mantissa with three endings, for both parities of the exponent
__device__ double value(unsigned top, int end, int e) {
    const unsigned long long low = end == 0 ? 0ull : end == 1 ? (1ull << 29) - 1 : (top * 2654435761ull) & ((1ull << 29) - 1);
    return __longlong_as_double(((1023ll + e) << 52) | ((unsigned long long)(top & 0x7fffff) << 29) | low);
}
__global__ void run(int op, unsigned long long* bad) {
    const unsigned long long tot = 6ull << 23;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < tot; i += (unsigned long long)gridDim.x * blockDim.x) {
        const double x = value((unsigned)(i & 0x7fffff), (int)((i >> 23) % 3), (int)(i / (3ull << 23)));
        bool ok = true;
        if (op) {
            ok = __double_as_longlong(lu::sqrt_int(x)) == __double_as_longlong(__dsqrt_rn(x));
        } else {
            const unsigned rec = lu::div_rec(x);
            const double a[4] = {1.0, __longlong_as_double(__double_as_longlong(x) - 1), x * 1.4142135623730951,
                                 __longlong_as_double((__double_as_longlong(x) * 6364136223846793005ll & 0xfffffffffffffll) | 0x3ff0000000000000ll)};
            for (int k = 0; k < 4; ++k)
                ok = ok && __double_as_longlong(lu::div_by(a[k], x, rec)) == __double_as_longlong(__ddiv_rn(a[k], x));
        }
        if (!ok) atomicAdd(bad, 1ull);
    }
}
extern "C" long long check_gpu(int op) {
    unsigned long long *d = nullptr, h = 0;
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return -1;
    run<<<1024, 256>>>(op, d);
    if (cudaGetLastError() != cudaSuccess || cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    cudaFree(d);
    return (long long)h;
}
"""


def _operands(seed, n):
    """Mantissas of all kinds: random, next to 1, 2 and the halves between
    doubles, exact quotients and squares and their neighbours."""
    r = np.random.default_rng(seed)
    m = 1.0 + r.random(n)
    near = r.integers(-40, 41, size=n)
    b = np.where(r.random(n) < 0.3, np.nextafter(np.where(r.random(n) < 0.5, 1.0, 2.0), 1.5) + near * 2.0 ** -52, m)
    b = np.clip(b, 1.0, np.nextafter(2.0, 0.0))
    q = 1.0 + np.floor(r.random(n) * 2.0 ** 26) * 2.0 ** -26
    a = np.where(r.random(n) < 0.4, (b.view(np.int64) & ~((1 << 27) - 1)).view(np.float64) * q, 1.0 + r.random(n))
    a = (a.view(np.int64) + r.integers(-2, 3, size=n)).view(np.float64)
    return a, b


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("ddiv")
    src, so = d / "host.cpp", d / "host.so"
    src.write_text(HOST)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", f"-I{CSRC}", f"-I{cuda}/include",
                    str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).check
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong] + [ctypes.c_void_p] * 3
    f.restype = ctypes.c_longlong
    return f


def _check(f, op, ulp, a, b):
    a, b, where = np.ascontiguousarray(a), np.ascontiguousarray(b), np.zeros(3)
    bad = f(op, ulp, a.size, a.ctypes.data, b.ctypes.data, where.ctypes.data)
    assert bad == 0, [float(v).hex() for v in where]


@pytest.mark.parametrize("ulp", [-1, 0, 1])
def test_division(host, ulp):
    a, b = _operands(1, 1 << 20)
    _check(host, 0, ulp, a, b)
    s = np.where(np.arange(a.size) % 2 == 0, 1.0, -1.0)
    _check(host, 0, ulp, np.ldexp(a * s, (np.arange(a.size) * 7) % 1800 - 900), np.ldexp(b, (np.arange(a.size) * 5) % 900 - 450))


@pytest.mark.parametrize("ulp", [-1, 0, 1])
def test_root(host, ulp):
    a, b = _operands(2, 1 << 20)
    e = np.arange(a.size) % 2
    _check(host, 1, ulp, np.ldexp(b, e), b)
    squares = a * a                            # and their neighbours
    _check(host, 1, ulp, (squares.view(np.int64) + np.arange(a.size) % 5 - 2).view(np.float64), b)
    top = np.nextafter(4.0, 0.0) - np.arange(1 << 16) * 2.0 ** -51
    _check(host, 1, ulp, top, top)
    _check(host, 1, ulp, np.ldexp(b, (np.arange(b.size) * 3) % 2000 - 1000), b)


@pytest.mark.parametrize("ulp", [-1, 0, 1])
def test_every_other_operand_goes_to_the_hardware(host, ulp):
    v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0.0),
                  np.finfo(float).max, 1.0, -3.0, 2.0 ** -600, 2.0 ** 700, 1.5 * 2.0 ** 1023])
    a, b = [x.ravel() for x in np.meshgrid(v, v)]
    _check(host, 0, ulp, a, b)
    _check(host, 1, ulp, v, v)


@pytest.mark.gpu
@pytest.mark.parametrize("op", [0, 1])
def test_on_the_gpu_over_every_input_of_the_approximations(tmp_path, op):
    from tests.gpu_util import cuda_or_fail
    cuda_or_fail()
    from paper_2010_05975_gb300 import build
    src, so = tmp_path / "gpu.cu", tmp_path / "gpu.so"
    src.write_text(GPU)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "--fmad=false", "-Xcompiler", "-fPIC", "-shared",
                    f"-I{CSRC}", str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).check_gpu
    f.argtypes, f.restype = [ctypes.c_int], ctypes.c_longlong
    assert f(op) == 0
