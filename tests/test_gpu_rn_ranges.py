"""The branch-free correctly rounded operations over the ranges they state, and the rotation of the shared tier's
columns-in-registers form against the built-in operations' over every range of norms and products."""
import ctypes
import importlib
import os
import subprocess

import pytest

from conftest import ROOT

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "jacobi_rx.cu"
using namespace bsvd;
__device__ unsigned long long bad[5];
__device__ void same(int i, float x, float y)
{
    if (__float_as_uint(x) != __float_as_uint(y) && !(isnan(x) && isnan(y))) atomicAdd(&bad[i], 1ull);
}
__device__ unsigned step(unsigned& s) { return s = s * 1664525u + 1013904223u; }
__global__ void operations()
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    const float m = __uint_as_float(0x3f800000u | (i & 0x7fffffu));
    for (int e = -100; e < 118; ++e) {
        const float x = ldexpf(m, e);
        if (e < 100) {
            same(0, rn_rcp(x), __frcp_rn(x));
            same(0, rn_rcp(-x), __frcp_rn(-x));
        }
        same(1, rn_sqrt(x), __fsqrt_rn(x));
    }
    unsigned s = i * 2654435761u + 12345u;
    for (int k = 0; k < 32; ++k) {
        const float mb = __uint_as_float(0x3f800000u | (step(s) >> 9));
        const int ea = int((step(s) >> 8) % 200u) - 100;
        int eb = int((step(s) >> 8) % 200u) - 100;
        eb = ea - eb > 98 ? ea - 98 : (ea - eb < -101 ? ea + 101 : eb);
        const float a = ldexpf(s & 1024u ? m : -m, ea), b = ldexpf(s & 2048u ? mb : -mb, eb);
        same(2, rn_div(a, b), __fdiv_rn(a, b));
    }
}
// a warp's operands: all inside the branch-free range, or anything
__global__ void rotations()
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned s = i * 2246822519u + 77u;
    for (int k = 0; k < 64; ++k) {
        const bool inside = ((i >> 5) + k) & 1;
        const float ma = __uint_as_float(0x3f800000u | (step(s) >> 9)), mb = __uint_as_float(0x3f800000u | (step(s) >> 9));
        const int span = inside ? 80 : 140;
        const int ea = int((step(s) >> 8) % (2u * span)) - span;
        const unsigned near = step(s) >> 28;   // the other norm: independent, close by, or a few last places away
        const int eb = near < 4 ? int((step(s) >> 8) % (2u * span)) - span : (near < 10 ? ea + int(near) - 7 : ea);
        float al = ldexpf(ma, ea), be = ldexpf(near < 10 ? mb : ma, eb);
        if (near == 15) be = __uint_as_float(__float_as_uint(be) + (step(s) >> 29));
        const double cosine = ldexp(double(mb), -int((step(s) >> 8) % 28u) - 1);
        float ga = float(sqrt(double(al) * double(be)) * cosine);
        if (s & 4096u) ga = -ga;
        if (!inside) {
            const unsigned odd = step(s) >> 24;
            const float inf = __int_as_float(0x7f800000), nan = __int_as_float(0x7fc00000);
            if (odd == 1) al = 0.f;
            if (odd == 2) be = inf;
            if (odd == 3) ga = nan;
            if (odd == 4) ga = 0.f;
            if (odd == 5) al = nan;
            if (odd == 6) ga = inf;
            if (odd == 7) be = -0.f;
        }
        const float tol = float(sqrt(128.0) * Unit<float>::value);
        float c, sn, c2 = 1.f, s2 = 0.f;
        const bool r = rx_rotation<float>(al, be, ga, tol, c, sn);
        const bool r2 = jacobi_rotation<float>(al, be, ga, tol, c2, s2);
        if (r != r2) atomicAdd(&bad[3], 1ull);
        same(4, c, r2 ? c2 : 1.f);
        same(4, sn, r2 ? s2 : 0.f);
    }
}
extern "C" int check(unsigned long long* out)
{
    operations<<<(1 << 23) / 256, 256>>>();
    rotations<<<1 << 13, 256>>>();
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    return cudaMemcpyFromSymbol(out, bad, sizeof(bad)) != cudaSuccess;
}
"""


def test_ranges(tmp_path):
    b = importlib.import_module("paper_1707_05141_gb300.build")
    src, so = tmp_path / "rn.cu", tmp_path / "librn.so"
    src.write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-I", b.CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(so)], check=True)
    out = (ctypes.c_ulonglong * 5)()
    assert ctypes.CDLL(str(so)).check(out) == 0
    assert list(out) == [0] * 5
