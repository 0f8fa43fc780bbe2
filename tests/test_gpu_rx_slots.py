"""GPU parity of the shared tier's columns-in-registers forms, each instance by the bound that selects it: the
edges of its slots, one slot, odd column counts, tall and wide, one factor alone; and the same numbers, bit for
bit, from every instance that can hold a matrix."""
import numpy as np
import pytest

from parity import gate, svd_errors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(bs, mats, bound, wide, want_u=True, want_v=True):
    if wide:
        mats = [a.T for a in mats]
    m, n = (np.array([a.shape[i] for a in mats], np.int32) for i in (0, 1))
    k = np.minimum(m, n)
    off = np.concatenate([[0], np.cumsum((m * n + 3) // 4 * 4)])
    flat = np.zeros(int(off[-1]) + 8, np.float32)
    for a, o in zip(mats, off):
        flat[o:o + a.size] = a.T.reshape(-1)
    A = bs.Batch.packed(torch.from_numpy(flat).cuda(), off[:-1], m, n)
    A.max_m, A.max_n = (bound, 128) if wide else (128, bound)
    ou, ov, os_ = (np.concatenate([[0], np.cumsum(x * k)]) for x in (m, n, np.ones_like(k)))
    fu, fv, fs = (torch.zeros(int(o[-1]), device="cuda") for o in (ou, ov, os_))
    info = torch.zeros(len(m), dtype=torch.int32, device="cuda")
    rot = torch.zeros(len(m), dtype=torch.int64, device="cuda")
    bs.batched_svd_jacobi(A, bs.Batch.packed(fs, os_[:-1], k, np.ones_like(k)),
                          bs.Batch.packed(fu, ou[:-1], m, k) if want_u else None,
                          bs.Batch.packed(fv, ov[:-1], n, k) if want_v else None, info, rot, tier=bs.TIER_SHARED)
    torch.cuda.synchronize()
    return mats, (fu, fv, fs, info, rot), (ou, ov, os_)


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("bound", [2, 9, 15, 16, 17, 32, 33, 48, 49, 64, 65, 95, 96, 97, 111, 112, 113, 128])
def test_instances(bound, wide):
    import paper_1707_05141_gb300 as bs
    bs.build()
    rng = np.random.default_rng(bound)
    shapes = [(128, bound), (bound, bound), (max(bound, 127), bound - 1), (128, 1), (1, 1), (2, 2), (max(bound, 5), min(bound, 3)),
              (max(bound, 66), (bound + 1) // 2)]
    mats = []
    for i, (m, n) in enumerate(shapes):
        a = rng.standard_normal((m, n)) * np.exp(-np.arange(n) / 8.0)
        if i == 2 and n > 3:
            a[:, 2] = a[:, 1]   # rank deficient
        mats.append(a.astype(np.float32))
    mats, out, (ou, ov, os_) = _run(bs, mats, bound, wide)
    hu, hv, hs, info, _ = (x.cpu().numpy() for x in out)
    for b, a in enumerate(mats):
        (m, n), k = a.shape, min(a.shape)
        assert 0 < info[b] < bs.INFO_NOT_CONVERGED, (a.shape, info[b])
        a64 = a.astype(np.float64)
        e = svd_errors(a64, hu[ou[b]:ou[b] + m * k].reshape(k, m).T, hs[os_[b]:os_[b] + k],
                       hv[ov[b]:ov[b] + n * k].reshape(k, n).T, np.linalg.svd(a64, compute_uv=False))
        names = ("sigma", "resid") if b == 2 else e   # (the vectors of a zero value are not unique)
        assert max(e[x] for x in names) <= gate(np.float32), (a.shape, e)
    back = [a.T for a in mats] if wide else mats
    for want in ((True, False), (False, True), (False, False)):   # one factor alone: the same numbers
        _, alone, _ = _run(bs, back, bound, wide, *want)
        for x, y, on in zip(alone, out, want + (True, True, True)):
            assert not on or torch.equal(x, y)
    _, largest, _ = _run(bs, back, 128, wide)   # the 64-slot instance
    for x, y in zip(largest, out):
        assert torch.equal(x, y)
