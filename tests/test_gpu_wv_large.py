"""GPU parity of the register tier's form with W and V in separate warps at the edges of its layout, in batches large
enough for every plain, carried, FP64-parameter and 128-row variant to take it; and the same numbers, bit for bit,
from a small batch, which takes the form with both in the same warps."""
import numpy as np
import pytest

from parity import gate, svd_errors
from test_gpu_wv import SHAPES64, SHAPES128, _batch

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (the form is taken beyond two to four matrices per SM)
PER_SM = 4


@pytest.fixture(scope="module")
def bs():
    import paper_1707_05141_gb300 as bs
    bs.build()
    return bs


def _variant(bs, m, n, carried=0, fp64=0, ctas=None):
    for k in range(1, bs.jacobi_variants(bs.F32, m, n, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(bs.F32, m, n, k)
        if (d["slots"], d["rows_a"], d["scaled"], d["qr_precond"], d["carried_norms"], d["fp64_params"]) == (
                32, 32, 1, 0, carried, fp64) and ctas in (None, d["ctas_per_sm"]):
            return bs.TIER_REGISTER | (k << 8)
    raise AssertionError((m, n, carried, fp64))


@pytest.mark.parametrize("pad,shift", [(0, 0), (3, 0), (4, 1)])
@pytest.mark.parametrize("form", ["64 plain", "64 carried", "64 FP64 parameters", "128 tall", "128 wide"])
def test_edges_in_large_batches(bs, form, pad, shift):
    if form.startswith("64"):
        kinds, bound = SHAPES64, (64, 64)
    elif form == "128 tall":
        kinds, bound = [s for s in SHAPES128 + SHAPES64 if s[0] >= s[1]], (128, 64)
    else:
        kinds, bound = [s for s in SHAPES128 + SHAPES64 if s[0] < s[1]], (64, 128)
    count = PER_SM * torch.cuda.get_device_properties(0).multi_processor_count + len(kinds)
    shapes = [kinds[i % len(kinds)] for i in range(count)]
    tier = _variant(bs, *bound, carried=int("carried" in form), fp64=int("FP64" in form))
    mats, A = _batch(bs, shapes, pad, shift, 11)
    A.max_m, A.max_n = bound
    m, n = (np.array([a.shape[i] for a in mats], np.int32) for i in (0, 1))
    k = np.minimum(m, n)
    ou, ov, os_ = (np.concatenate([[0], np.cumsum((x + 3) // 4 * 4)]) for x in ((m + pad) * k + 4, (n + pad) * k + 4, k))

    def run(want_u, want_v):
        fu, fv, fs = (torch.zeros(int(o[-1]) + shift + 8, device="cuda") for o in (ou, ov, os_))
        info = torch.zeros(count, dtype=torch.int32, device="cuda")
        bs.batched_svd_jacobi(A, bs.Batch.packed(fs, os_[:-1], k, np.ones_like(k)),
                              bs.Batch.packed(fu, ou[:-1] + shift, m, k, m + pad) if want_u else None,
                              bs.Batch.packed(fv, ov[:-1] + shift, n, k, n + pad) if want_v else None, info, tier=tier)
        torch.cuda.synchronize()
        return fu, fv, fs, info

    out = run(True, True)
    for want in ((True, False), (False, True), (False, False)):
        for x, y, on in zip(run(*want), out, want + (True, True)):
            assert not on or torch.equal(x, y)
    hu, hv, hs, hi = (x.cpu().numpy() for x in out)
    for b, a in enumerate(mats):
        take = lambda f, o, r: np.stack([f[o + shift + c * (r + pad):][:r] for c in range(k[b])], 1)  # noqa: E731
        assert 0 < hi[b] < bs.INFO_NOT_CONVERGED, (a.shape, hi[b])
        a64 = a.astype(np.float64)
        e = svd_errors(a64, take(hu, ou[b], m[b]), hs[os_[b]:os_[b] + k[b]], take(hv, ov[b], n[b]),
                       np.linalg.svd(a64, compute_uv=False))
        assert max(e.values()) <= gate(np.float32), (a.shape, e)


@pytest.mark.parametrize("m,n,want", [(64, 64, {}), (54, 45, {}), (37, 64, {}), (54, 45, dict(ctas=4)), (120, 50, {}),
                                      (64, 100, {}), (64, 64, dict(carried=1)), (54, 45, dict(carried=1)),
                                      (33, 60, dict(carried=1)), (64, 64, dict(fp64=1)), (40, 33, dict(fp64=1))])
def test_both_forms_agree(bs, m, n, want):
    small = torch.cuda.get_device_properties(0).multi_processor_count   # one matrix per SM
    large = PER_SM * small + 1
    tier = _variant(bs, m, n, **want)
    a = torch.randn((large, n, m), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    a *= torch.exp(-torch.arange(n, device="cuda") / 8.0)[None, :, None]
    k = min(m, n)

    def run(x):
        b = x.shape[0]
        s, u, v = (torch.zeros(z, device="cuda") for z in ((b, 1, k), (b, k, m), (b, k, n)))
        info = torch.zeros(b, dtype=torch.int32, device="cuda")
        rot = torch.zeros(b, dtype=torch.int64, device="cuda")
        bs.batched_svd_jacobi(bs.Batch.uniform(x, m, n), bs.Batch.uniform(s, k, 1), bs.Batch.uniform(u, m, k),
                              bs.Batch.uniform(v, n, k), info, rot, tier=tier)
        return s, u, v, info, rot

    one = run(a)
    parts = [run(x.contiguous()) for x in a.split(small)]
    for i, x in enumerate(one):
        assert torch.equal(x, torch.cat([p[i] for p in parts]))
