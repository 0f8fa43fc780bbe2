"""GPU parity of the shared tier's columns-in-registers form at the edges of its slots: one to 64 of them, odd
column counts, wide matrices, unaligned storage, values only, one side only, norms past the range of its
branch-free parameters."""
import numpy as np
import pytest

from parity import gate, svd_errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 1), (2, 2), (3, 3), (4, 4), (5, 3), (64, 2), (65, 65), (96, 33), (127, 100), (100, 127), (128, 127),
          (127, 128), (128, 128), (2, 128), (1, 128), (128, 1), (66, 34)]


# (the small scale has no decay and no dependent columns: their squared norms would be FP32 denormals)
@pytest.mark.parametrize("scale,decay,dependent", [(1.0, 8.0, True), (1e-16, np.inf, False), (1e16, 8.0, True)])
def test_edges_of_the_slots(scale, decay, dependent):
    import paper_1707_05141_gb300 as bs
    bs.build()
    rng = np.random.default_rng(3)
    m, n = (np.array([s[i] for s in SHAPES], np.int32) for i in (0, 1))
    k = np.minimum(m, n)
    mats = []
    for i, (mm, nn) in enumerate(SHAPES):
        a = rng.standard_normal((mm, nn)) * np.exp(-np.arange(nn) / decay)
        if dependent and i % 3 == 2 and nn > 3:
            a[:, 1] = a[:, 0]   # rank deficient
            a[:, 2] = 0
        mats.append((a * scale).astype(np.float32))
    ld = m + 1
    off = np.concatenate([[0], np.cumsum((ld * n + 3) // 4 * 4)]) + 1
    flat = np.full(int(off[-1]) + 8, 5.0, np.float32)
    for a, o, l in zip(mats, off, ld):
        for j in range(a.shape[1]):
            flat[o + j * l:o + j * l + a.shape[0]] = a[:, j]
    A = bs.Batch.packed(torch.from_numpy(flat).cuda(), off[:-1], m, n, ld)
    ou, ov, os_ = (np.concatenate([[0], np.cumsum(x * k + 4)]) for x in (m, n, np.ones_like(k)))

    def run(want_u, want_v):
        fu, fv, fs = (torch.zeros(int(o[-1]) + 8, device="cuda") for o in (ou, ov, os_))
        info = torch.zeros(len(m), dtype=torch.int32, device="cuda")
        bs.batched_svd_jacobi(A, bs.Batch.packed(fs, os_[:-1], k, np.ones_like(k)),
                              bs.Batch.packed(fu, ou[:-1], m, k) if want_u else None,
                              bs.Batch.packed(fv, ov[:-1], n, k) if want_v else None, info, tier=bs.TIER_SHARED)
        torch.cuda.synchronize()
        return fu, fv, fs, info.cpu().numpy()

    fu, fv, fs, info = run(True, True)
    for want in ((False, False), (True, False), (False, True)):
        gu, gv, gs, _ = run(*want)
        assert torch.equal(gs, fs)
        assert not want[0] or torch.equal(gu, fu)
        assert not want[1] or torch.equal(gv, fv)
    hu, hv, hs = (x.cpu().numpy().astype(np.float64) for x in (fu, fv, fs))
    for b, a in enumerate(mats):
        assert 0 < info[b] < bs.INFO_NOT_CONVERGED, (a.shape, info[b])
        a64 = a.astype(np.float64)
        u = hu[ou[b]:ou[b] + m[b] * k[b]].reshape(k[b], m[b]).T
        v = hv[ov[b]:ov[b] + n[b] * k[b]].reshape(k[b], n[b]).T
        s = hs[os_[b]:os_[b] + k[b]]
        ref = np.linalg.svd(a64, compute_uv=False)
        e = svd_errors(a64, u, s, v, ref)
        if dependent and b % 3 == 2 and a.shape[1] > 3:   # the vectors of the zero values are not unique
            assert max(e["sigma"], e["resid"]) <= gate(np.float32), (a.shape, e)
        else:
            assert max(e.values()) <= gate(np.float32), (a.shape, e)
