"""GPU parity of the register tier's form with W and V in separate warps (32 slots, 64 or 128 rows) at the
edges of its layout, and of the branch-free correctly rounded operations it computes its parameters with."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT
from parity import gate, svd_errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bs():
    import paper_1707_05141_gb300 as bs
    bs.build()
    assert torch.cuda.is_available()
    return bs


def _batch(bs, shapes, pad, shift, seed):
    """Column-major matrices of ``shapes`` with leading dimension rows + pad, the storage shifted by
    ``shift`` elements (0 and 0: 16-byte aligned columns for rows a multiple of 4)."""
    rng = np.random.default_rng(seed)
    mats = []
    for m, n in shapes:
        k = max(1, min(m, n))
        u, _ = np.linalg.qr(rng.standard_normal((m, k)))
        v, _ = np.linalg.qr(rng.standard_normal((n, k)))
        mats.append(((u * np.exp(-np.arange(u.shape[1]) / 8.0)) @ v.T).astype(np.float32))
    ld = [m + pad for m, _ in shapes]
    size = [(l * n + 7) // 4 * 4 for l, (_, n) in zip(ld, shapes)]
    off = np.concatenate([[0], np.cumsum(size)[:-1]]) + shift
    flat = np.full(int(sum(size)) + shift + 8, 7.0, np.float32)
    for a, o, l in zip(mats, off, ld):
        for j in range(a.shape[1]):
            flat[o + j * l:o + j * l + a.shape[0]] = a[:, j]
    t = torch.from_numpy(flat).cuda()
    m, n = (np.array([s[i] for s in shapes], np.int32) for i in (0, 1))
    return mats, bs.Batch.packed(t, off, m, n, np.array(ld, np.int32))


SHAPES64 = [(1, 1), (2, 1), (3, 3), (5, 4), (31, 31), (32, 32), (33, 33), (40, 63), (63, 64), (64, 63), (64, 1), (64, 64)]
SHAPES128 = [(65, 64), (96, 33), (127, 63), (128, 64), (64, 128), (66, 66 - 2), (1, 128), (128, 2)]


@pytest.mark.parametrize("pad,shift", [(0, 0), (3, 0), (4, 1)])
@pytest.mark.parametrize("bound", ["64 plain", "64 carried", "64 preconditioned", "64 FP64 parameters", "128"])
def test_edges_of_the_layout(bs, bound, pad, shift):
    big = bound == "128"
    shapes = SHAPES128 if big else SHAPES64
    mats, A = _batch(bs, shapes, pad, shift, 11)
    max_m, max_n = (128, 64) if big else (64, 64)
    variant = 0
    for k in range(1, bs.jacobi_variants(bs.F32, max_m, max_n, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(bs.F32, max_m, max_n, k)
        want = dict(qr_precond=int("precond" in bound), fp64_params=int("FP64" in bound),
                    carried_norms=int("carried" in bound or "precond" in bound))
        if d["slots"] == 32 and all(d[x] == y for x, y in want.items()):
            variant = variant or k
    A.max_m, A.max_n = (128, 128) if big else (64, 64)
    if big:
        # wide and tall matrices together are bounded by 128 x 128, past the register tier: two calls
        sel = [[i for i, (m, n) in enumerate(shapes) if m >= n], [i for i, (m, n) in enumerate(shapes) if m < n]]
    else:
        sel = [list(range(len(shapes)))]
    for idx in sel:
        mats, A = _batch(bs, [shapes[i] for i in idx], pad, shift, 11)
        m = np.array([a.shape[0] for a in mats], np.int32)
        n = np.array([a.shape[1] for a in mats], np.int32)
        k = np.minimum(m, n)
        if big:
            A.max_m, A.max_n = (128, 64) if m[0] >= n[0] else (64, 128)
        else:
            A.max_m, A.max_n = 64, 64
        su, sv = (m + pad) * k + 4, (n + pad) * k + 4
        ou, ov, os_ = (np.concatenate([[0], np.cumsum((x + 3) // 4 * 4)]) for x in (su, sv, k))
        fu, fv, fs = (torch.zeros(int(o[-1]) + shift + 8, device="cuda") for o in (ou, ov, os_))
        U = bs.Batch.packed(fu, ou[:-1] + shift, m, k, m + pad)
        V = bs.Batch.packed(fv, ov[:-1] + shift, n, k, n + pad)
        S = bs.Batch.packed(fs, os_[:-1], k, np.ones_like(k))
        info = torch.zeros(len(m), dtype=torch.int32, device="cuda")
        bs.batched_svd_jacobi(A, S, U, V, info, tier=bs.TIER_REGISTER | (variant << 8))
        torch.cuda.synchronize()
        hu, hv, hs, hi = fu.cpu().numpy(), fv.cpu().numpy(), fs.cpu().numpy(), info.cpu().numpy()
        # values only, and one side only: the same numbers
        fs2, fv2 = torch.zeros_like(fs), torch.zeros_like(fv)
        S2 = bs.Batch.packed(fs2, os_[:-1], k, np.ones_like(k))
        V2 = bs.Batch.packed(fv2, ov[:-1] + shift, n, k, n + pad)
        bs.batched_svd_jacobi(A, S2, None, None, info, tier=bs.TIER_REGISTER | (variant << 8))
        assert torch.equal(fs2, fs)
        bs.batched_svd_jacobi(A, S2, None, V2, info, tier=bs.TIER_REGISTER | (variant << 8))
        assert torch.equal(fs2, fs) and torch.equal(fv2, fv)
        for b, a in enumerate(mats):
            a64 = a.astype(np.float64)
            take = lambda f, o, r: np.stack([f[o + shift + c * (r + pad):][:r] for c in range(k[b])], 1)  # noqa: E731
            assert 0 < hi[b] < bs.INFO_NOT_CONVERGED, (a.shape, hi[b])
            e = svd_errors(a64, take(hu, ou[b], m[b]), hs[os_[b]:os_[b] + k[b]], take(hv, ov[b], n[b]),
                           np.linalg.svd(a64, compute_uv=False))
            assert max(e.values()) <= gate(np.float32), (a.shape, e)


SOURCE = r"""
#include "rnmath.cuh"
using namespace bsvd;
__device__ unsigned long long bad[4];
__global__ void every_mantissa()
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    const float m = __uint_as_float(0x3f800000u | (i & 0x7fffffu));
    for (int e = -40; e <= 3; ++e) {
        const float x = ldexpf(m, e);
        if (__float_as_uint(rn_rcp(x)) != __float_as_uint(__frcp_rn(x))) atomicAdd(&bad[0], 1ull);
        if (__float_as_uint(rn_sqrt(x)) != __float_as_uint(__fsqrt_rn(x))) atomicAdd(&bad[1], 1ull);
    }
    if (__float_as_uint(rn_rsqrt12(m)) != __float_as_uint(__frsqrt_rn(m))) atomicAdd(&bad[2], 1ull);
    // quotients: this mantissa against 16 pseudo-random divisors, the largest mantissas among them
    unsigned s = i * 2654435761u + 12345u;
    for (int k = 0; k < 16; ++k) {
        s = s * 1664525u + 1013904223u;
        const float b = ldexpf(__uint_as_float(k == 0 ? 0x3fffffffu : 0x3f800000u | (s >> 9)), k % 3);
        const float a = ldexpf(k & 1 ? -m : m, -(int)(s % 97u));
        if (__float_as_uint(rn_div(a, b)) != __float_as_uint(__fdiv_rn(a, b))) atomicAdd(&bad[3], 1ull);
    }
}
extern "C" int rn_check(unsigned long long* out)
{
    every_mantissa<<<(1 << 23) / 256, 256>>>();
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    return cudaMemcpyFromSymbol(out, bad, sizeof(bad)) != cudaSuccess;
}
"""


def test_branch_free_operations_are_correctly_rounded(tmp_path):
    """Every mantissa of the reciprocal, square root and reciprocal square root, 2^27 quotients."""
    import importlib
    b = importlib.import_module("paper_1707_05141_gb300.build")
    src, so = tmp_path / "rn.cu", tmp_path / "librn.so"
    src.write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", b.CSRC,
                    "-I", os.path.join(ROOT, "include"), str(src), "-o", str(so)], check=True)
    out = (ctypes.c_ulonglong * 4)()
    assert ctypes.CDLL(str(so)).rn_check(out) == 0
    assert list(out) == [0, 0, 0, 0]


@pytest.mark.parametrize("vectors", [True, False])
@pytest.mark.parametrize("m,n,carried", [(54, 45, False), (64, 64, True), (37, 64, False), (120, 50, False)])
def test_small_and_large_batches_agree(bs, m, n, carried, vectors):
    """The plain 32-slot variants take a batch of more than two matrices per SM to the form with W and V in
    separate warps and a smaller one to the form with both in the same: the same numbers, bit for bit."""
    per = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    variant = 0
    for k in range(1, bs.jacobi_variants(bs.F32, m, n, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(bs.F32, m, n, k)
        if carried and d["carried_norms"] and not d["qr_precond"] and d["slots"] == 32:
            variant = k
    assert bool(variant) == carried
    a = torch.randn((per + 1, n, m), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    a *= torch.exp(-torch.arange(n, device="cuda") / 8.0)[None, :, None]
    k = min(m, n)

    def run(x):
        b = x.shape[0]
        s, u, v = (torch.zeros(z, device="cuda") for z in ((b, 1, k), (b, k, m), (b, k, n)))
        info = torch.zeros(b, dtype=torch.int32, device="cuda")
        rot = torch.zeros(b, dtype=torch.int64, device="cuda")
        U = bs.Batch.uniform(u, m, k) if vectors else None
        V = bs.Batch.uniform(v, n, k) if vectors else None
        bs.batched_svd_jacobi(bs.Batch.uniform(x, m, n), bs.Batch.uniform(s, k, 1), U, V, info, rot,
                              tier=bs.TIER_REGISTER | (variant << 8))
        return s, u, v, info, rot

    large, small, last = run(a), run(a[:per].contiguous()), run(a[per:].contiguous())
    for x, y, z in zip(large, small, last):
        assert torch.equal(x, torch.cat([y, z]))
