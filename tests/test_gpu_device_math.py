"""The device helpers that decide statuses and pivots on a fast path, against the plain expressions
they replace, on the GPU (a small library of its own is compiled from the header).

lp_rcp(float): bit for bit the correctly rounded reciprocal, over all 2^32 inputs.
lp_rcp(double): the seed's relative error is below 2^-22 (truncation to float32 and an
approximation within one ulp), so the cubic step leaves 2^-66 and its inner roundings 2^-73: within
half an ulp and 2^-13 of one, that is at most one ulp from the rounded quotient, in at most
2^-11 of all cases (a bound of 2^-10 here).
within, pivot_vanished: the same decision as the exact test, everywhere.
"""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2503_13075_gb300 import build  # noqa: E402

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "devmath.cuh"
using namespace ilves;
struct Mode { static constexpr double pivot_rel = 1e-13; };
__global__ void k_rcp32(unsigned long long* bad) {
    unsigned long long n = 0;
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += gridDim.x * blockDim.x) {
        const float a = __uint_as_float((unsigned)i), x = lp_rcp(a), y = __frcp_rn(a);
        n += __float_as_uint(x) != __float_as_uint(y) && !(x != x && y != y);
    }
    atomicAdd(bad, n);
}
__global__ void k_rcp64(const double* a, int n, double* fast, double* ref) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { fast[i] = lp_rcp(a[i]); ref[i] = __drcp_rn(a[i]); }
}
__global__ void k_within(const double* s, const double* tol, const double* d2, int n, int* got, int* want) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { got[i] = within(s[i], tol[i], d2[i]); want[i] = fabs(s[i]) <= tol[i] * d2[i]; }
}
__global__ void k_pivot(const double* s, const double* a, int n, int* got, int* want) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { got[i] = pivot_vanished<Mode>(s[i], a[i]); want[i] = !(fabs(s[i]) > Mode::pivot_rel * fabs(a[i])); }
}
extern "C" int rcp32(void* bad) { k_rcp32<<<1216, 256>>>((unsigned long long*)bad); return (int)cudaDeviceSynchronize(); }
extern "C" int rcp64(void* a, int n, void* f, void* r) {
    k_rcp64<<<(n + 255) / 256, 256>>>((double*)a, n, (double*)f, (double*)r); return (int)cudaDeviceSynchronize(); }
extern "C" int within_(void* s, void* t, void* d, int n, void* g, void* w) {
    k_within<<<(n + 255) / 256, 256>>>((double*)s, (double*)t, (double*)d, n, (int*)g, (int*)w); return (int)cudaDeviceSynchronize(); }
extern "C" int pivot(void* s, void* a, int n, void* g, void* w) {
    k_pivot<<<(n + 255) / 256, 256>>>((double*)s, (double*)a, n, (int*)g, (int*)w); return (int)cudaDeviceSynchronize(); }
"""


@pytest.fixture(scope="module")
def math(tmp_path_factory):
    d = tmp_path_factory.mktemp("devmath")
    (d / "m.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, "-shared", "-Xcompiler", "-fPIC",
                    str(d / "m.cu"), "-o", str(d / "m.so")], check=True)
    torch.cuda.init()
    return ctypes.CDLL(str(d / "m.so"))


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def any_double(rng, n):
    """Random bit patterns (every exponent alike, subnormals, infinities and NaN among them)."""
    return rng.integers(0, 1 << 64, n, dtype=np.uint64).view(np.float64)


def test_reciprocal_float(math):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    assert math.rcp32(ptr(bad)) == 0 and bad.item() == 0


def test_reciprocal_double(math):
    rng = np.random.default_rng(1)
    n = 1 << 22
    mid = (1 + rng.random(n)) * 2.0 ** rng.integers(-122, 123, n) * rng.choice([-1.0, 1.0], n)
    a = np.concatenate([mid, any_double(rng, n), [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1.0, 2.0**-1022, 2.0**1023]])
    da, f, r = dev(a), torch.empty(len(a), dtype=torch.float64, device="cuda"), torch.empty(len(a), dtype=torch.float64, device="cuda")
    assert math.rcp64(ptr(da), len(a), ptr(f), ptr(r)) == 0
    f, r = f.cpu().numpy(), r.cpu().numpy()
    same = (f == r) & (np.signbit(f) == np.signbit(r)) | (np.isnan(f) & np.isnan(r))
    off = np.abs(f[~same].view(np.int64) - r[~same].view(np.int64))
    assert off.max(initial=0) <= 1 and np.count_nonzero(~same[:n]) <= n * 2.0**-10


def test_within(math):
    rng = np.random.default_rng(2)
    n = 1 << 22
    d2 = 10.0 ** rng.uniform(-6, 2, n)
    tol = rng.choice([1e-12, 1e-8, 1e-4, 1e-16, 0.0, 1e-30, 1e-42, 1e-300, 0.3, 1e30, np.inf], n)
    step = rng.choice([0.0, 2.0**-52, 2.0**-40, 2.0**-24, 2.0**-22, 2.0**-21, 2.0**-20, 2.0**-19, 2.0**-10, 0.5], n)
    with np.errstate(all="ignore"):
        s = tol * d2 * (1 + step * rng.choice([-1.0, -0.99, 0.99, 1.0], n)) * rng.choice([-1.0, 1.0], n)
    wild = [any_double(rng, n), rng.choice(tol, n), d2]
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 1e-12, 1e300])
    e = [np.repeat(edge, 4), np.tile([0.0, 1e-12, 1e-300, 1.0], len(edge)), np.full(4 * len(edge), 0.01)]
    big = [rng.normal(size=1000) * 1e190, np.full(1000, 1e-12), np.full(1000, 1e200)]
    s, tol, d2 = (np.concatenate(v) for v in zip([s, tol, d2], wild, e, big))
    g, w = (torch.zeros(len(s), dtype=torch.int32, device="cuda") for _ in range(2))
    assert math.within_(ptr(dev(s)), ptr(dev(tol)), ptr(dev(d2)), len(s), ptr(g), ptr(w)) == 0
    assert torch.equal(g, w) and 0 < int(w.sum()) < len(s)


def test_pivot_vanished(math):
    rng = np.random.default_rng(3)
    n = 1 << 22
    a = 10.0 ** rng.uniform(-20, 20, n) * rng.choice([-1.0, 1.0], n)
    ratio = rng.choice([1e-13, 2.0**-43, 2.0**-42, 2.0**-44, 1e-3, 1.0, 1e5, 0.0], n)
    s = a * ratio * (1 + rng.choice([0.0, 2.0**-52, 2.0**-30, 0.3, 0.9], n) * rng.choice([-1.0, 1.0], n))
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0**-1022, 1.0, 1e300])
    s = np.concatenate([s, any_double(rng, n), np.repeat(edge, len(edge))])
    a = np.concatenate([a, any_double(rng, n), np.tile(edge, len(edge))])
    g, w = (torch.zeros(len(s), dtype=torch.int32, device="cuda") for _ in range(2))
    assert math.pivot(ptr(dev(s)), ptr(dev(a)), len(s), ptr(g), ptr(w)) == 0
    assert torch.equal(g, w) and 0 < int(w.sum()) < len(s)
