"""GPU parity of the blocked one-CTA QR (FP32, 32-column panels in registers) at the edges of its panels, row
registers, row vectors and column chunks, ragged batches, partial outputs and refused shapes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GATE = 1e-5   # the FP32 gate of the batched QR


@pytest.fixture(scope="module")
def bs():
    import paper_1707_05141_gb300 as bs
    bs.build()
    return bs


SHAPES = {
    (160, 128): [(128, 128), (127, 127), (65, 65), (97, 96), (33, 33), (160, 1), (1, 1), (64, 64), (100, 0), (50, 31)],
    (256, 150): [(256, 150), (250, 149), (255, 129), (150, 150), (131, 130), (253, 32), (161, 160 - 10), (40, 33)],
    (512, 70): [(512, 70), (511, 65), (509, 64), (70, 70), (257, 66), (300, 33), (512, 1)],
    (250, 170): [(250, 161), (169, 169), (249, 170), (193, 160)],
    (257, 48): [(257, 48), (48, 48), (256, 33), (63, 47)],
}


@pytest.mark.parametrize("bound", sorted(SHAPES))
@pytest.mark.parametrize("pad", [0, 3])
def test_edges(bs, bound, pad):
    rng = np.random.default_rng(7)
    mats = [rng.standard_normal(s).astype(np.float32) for s in SHAPES[bound]]
    mats[0][:, 1:2] = 0                       # a zero column
    if mats[1].shape[1] > 3:
        mats[1][:, 3] = mats[1][:, 2]         # a repeated one
    mats[2] *= np.float32(1e-12)
    b = len(mats)
    m, n = (np.array([a.shape[i] for a in mats], np.int32) for i in (0, 1))
    lda, ldq, ldr = m + pad, m + pad, n + pad + 1

    def flat(ld):
        off = np.concatenate([[0], np.cumsum(ld * np.maximum(n, 1))])
        return np.full(int(off[-1]) + 4, 9.0, np.float32), off[:-1]

    fa, oa = flat(lda)
    for a, o, l in zip(mats, oa, lda):
        for j in range(a.shape[1]):
            fa[o + j * l:o + j * l + a.shape[0]] = a[:, j]
    (fq, oq), (fr, orr) = flat(ldq), flat(ldr)
    ta, tq, tr = (torch.from_numpy(x).cuda() for x in (fa, fq, fr))
    info = torch.full((b,), 7, dtype=torch.int32, device="cuda")

    def batch(t, off, rows, cols, ld):
        x = bs.Batch.packed(t, off, rows, cols, ld)
        x.max_m, x.max_n = (bound if rows is m else (bound[1], bound[1]))
        return x

    A, Qb, Rb = batch(ta, oa, m, n, lda), batch(tq, oq, m, n, ldq), batch(tr, orr, n, n, ldr)
    bs.batched_qr(A, Qb, Rb, info)
    torch.cuda.synchronize()
    assert info.tolist() == [0] * b
    q, r = tq.cpu().numpy(), tr.cpu().numpy()
    used_q, used_r = np.zeros(q.size, bool), np.zeros(r.size, bool)
    for i, a in enumerate(mats):
        mm, nn = a.shape
        iq = oq[i] + np.arange(nn)[None, :] * ldq[i] + np.arange(mm)[:, None]
        ir = orr[i] + np.arange(nn)[None, :] * ldr[i] + np.arange(nn)[:, None]
        used_q[iq], used_r[ir] = True, True
        if nn == 0:
            continue
        qq, rr = q[iq].astype(np.float64), r[ir].astype(np.float64)
        assert np.abs(qq.T @ qq - np.eye(nn)).max() <= GATE
        assert np.linalg.norm(qq @ rr - a) <= GATE * max(np.linalg.norm(a), 1e-30)
        assert not np.tril(rr, -1).any()
    assert (q[~used_q] == 9.0).all() and (r[~used_r] == 9.0).all()   # nothing else is written
    # R alone, Q alone: the same numbers
    for only in ("q", "r"):
        t2q, t2r = torch.full_like(tq, 9.0), torch.full_like(tr, 9.0)
        bs.batched_qr(A, batch(t2q, oq, m, n, ldq) if only == "q" else None,
                      batch(t2r, orr, n, n, ldr) if only == "r" else None, info)
        assert torch.equal(t2q, tq) if only == "q" else torch.equal(t2r, tr)


def test_refused_shapes_and_nonfinite(bs):
    m, n = np.array([130, 60, 200, 130], np.int32), np.array([100, 61, 100, 100], np.int32)
    off = np.arange(4) * 20000
    t = torch.randn(80000, device="cuda")
    t[3 * 20000 + 5] = float("nan")
    A = bs.Batch.packed(t, off, m, n)
    A.max_m, A.max_n = 150, 100
    info = torch.zeros(4, dtype=torch.int32, device="cuda")
    q, r = torch.full((80000,), 9.0, device="cuda"), torch.full((80000,), 9.0, device="cuda")
    bs.batched_qr(A, bs.Batch.packed(q, off, m, n), bs.Batch.packed(r, off, n, n), info)
    assert info.tolist() == [0, bs.INFO_BAD_SHAPE, bs.INFO_BAD_SHAPE, bs.INFO_NONFINITE]
    assert (q[20000:60000] == 9.0).all() and (r[20000:60000] == 9.0).all()
