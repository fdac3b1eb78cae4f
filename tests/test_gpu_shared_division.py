"""``SharedDiv`` by itself against IEEE division (NumPy's): random operands,
quotients next to the midpoint of two numbers, and the ends of the ranges that
the method takes (significands just short of 2, the smallest and largest
divisors and numerators, zeros of either sign), in both widths. What it does not
take, it must refuse."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "lbm_div.cuh"
template <typename R>
__global__ void k(const R *a, const R *b, R *q, unsigned char *taken, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const lbm::SharedDiv<R> d(b[i]);
    const bool ok = d.ok && lbm::SharedDiv<R>::fits(a[i]);
    taken[i] = ok;
    q[i] = ok ? d.quot(a[i]) : R(0);
}
template <typename R>
static int run(const R *a, const R *b, R *q, unsigned char *taken, int n)
{
    char *m = nullptr;
    const size_t s = sizeof(R) * (size_t)n;
    if (cudaMalloc(&m, 3 * s + n) != cudaSuccess) return 1;
    R *da = (R *)m, *db = da + n, *dq = db + n;
    unsigned char *dt = (unsigned char *)(dq + n);
    cudaMemcpy(da, a, s, cudaMemcpyHostToDevice);
    cudaMemcpy(db, b, s, cudaMemcpyHostToDevice);
    k<R><<<(n + 255) / 256, 256>>>(da, db, dq, dt, n);
    cudaMemcpy(q, dq, s, cudaMemcpyDeviceToHost);
    const int rc = cudaMemcpy(taken, dt, n, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(m);
    return rc;
}
extern "C" int run32(const float *a, const float *b, float *q, unsigned char *t, int n) { return run(a, b, q, t, n); }
extern "C" int run64(const double *a, const double *b, double *q, unsigned char *t, int n) { return run(a, b, q, t, n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2303_02210_gb300 import build
    d = tmp_path_factory.mktemp("div")
    src, so = str(d / "div.cu"), str(d / "div.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    src, "-o", so], check=True)
    return ctypes.CDLL(so)


def operands(dtype):
    p, top, blo, bhi, alo, ahi = (24, 0x7FFF00, -30, 30, -60, 60) if dtype is np.float32 else \
        (53, 0xFE000 << 32, -100, 100, -500, 500)
    rng = np.random.default_rng(5)
    n = 1 << 20
    one = 1 << (p - 1)
    # divisors and numerators over the whole ranges
    mb, ma = (rng.integers(one, 2 * one, n).astype(np.float64) for _ in range(2))
    sb = np.ldexp(mb.astype(dtype) / dtype(one), rng.integers(blo, bhi, n)).astype(dtype)
    sa = np.ldexp(ma.astype(dtype) / dtype(one), rng.integers(alo, ahi, n)).astype(dtype) * rng.choice([-1, 1], n).astype(dtype)
    a, b = [sa], [sb]
    # quotients next to a midpoint: numerators rounded from b (q + half a unit)
    q = (rng.integers(one, 2 * one, n).astype(np.longdouble) + np.longdouble(0.5)) / np.longdouble(one)
    a.append((sb.astype(np.longdouble) * q).astype(dtype))
    b.append(sb)
    # the same by divisors just short of 2 (times a power of two)
    near = np.ldexp((one + rng.integers(top - (1 << (p - 7)), top, n)).astype(dtype) / dtype(one),
                    rng.integers(blo, bhi, n)).astype(dtype)
    a.append((near.astype(np.longdouble) * q).astype(dtype))
    b.append(near)
    # edges
    edge_b = [np.ldexp(dtype(one + m) / dtype(one), e).astype(dtype) for e in (blo, -1, 0, bhi - 1)
              for m in (0, 1, top - 2, top - 1, top, top + 1, one - 1)]
    edge_b += [np.ldexp(dtype(1), bhi).astype(dtype), np.nextafter(np.ldexp(dtype(1), blo).astype(dtype), dtype(0)),
               dtype(0), dtype(-1.5), dtype(np.inf), dtype(np.nan)]
    edge_a = [np.ldexp(dtype(1), alo).astype(dtype), np.nextafter(np.ldexp(dtype(1), alo).astype(dtype), dtype(0)),
              np.nextafter(np.ldexp(dtype(1), ahi).astype(dtype), dtype(0)), np.ldexp(dtype(1), ahi).astype(dtype),
              dtype(0), dtype(1), np.finfo(dtype).tiny, np.finfo(dtype).smallest_subnormal, dtype(np.inf), dtype(np.nan)]
    edge_a = edge_a + [-x for x in edge_a]
    ga, gb = np.meshgrid(np.array(edge_a, dtype), np.array(edge_b, dtype))
    a.append(ga.ravel())
    b.append(gb.ravel())
    a, b = np.concatenate(a), np.concatenate(b)
    bits = b.view(np.uint32 if p == 24 else np.uint64) & (one - 1)
    mag = np.abs(a)
    with np.errstate(invalid="ignore"):
        takes = (bits < top) & (b >= dtype(2.0 ** blo)) & (b < dtype(2.0 ** bhi)) & (
            (mag == 0) | ((mag >= dtype(2.0 ** alo)) & (mag < dtype(2.0 ** ahi))))
    return a, b, takes


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_quotients_are_ieee(lib, dtype):
    a, b, takes = operands(dtype)
    q = np.empty_like(a)
    taken = np.empty(a.size, np.uint8)
    fn = lib.run32 if dtype is np.float32 else lib.run64
    p = ctypes.c_void_p
    assert fn(p(a.ctypes.data), p(b.ctypes.data), p(q.ctypes.data), p(taken.ctypes.data), a.size) == 0
    assert np.array_equal(taken.astype(bool), takes)
    assert takes.sum() > 2.9e6
    u = np.uint32 if dtype is np.float32 else np.uint64
    assert np.array_equal(q[takes].view(u), (a[takes] / b[takes]).view(u))
