"""GPU parity: the blocked QR at the edges of its panels (rows per lane, CTAs per cluster) and of its block
reflectors (row slabs, column tiles), ragged batches with unaligned storage included."""
import numpy as np
import pytest

from parity import gate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES32 = [[(128, 33), (127, 32), (33, 33), (1, 1)], [(129, 65), (256, 64), (257, 31)], [(512, 40), (511, 33)],
            [(513, 64), (40, 40), (512, 1)], [(1025, 70), (1024, 65), (600, 64)], [(2049, 33), (2048, 96), (90, 64)],
            [(4097, 33), (4096, 32), (500, 33)], [(8200, 33), (300, 2)]]
SHAPES64 = [[(127, 33), (128, 64), (1, 1)], [(385, 40), (384, 33), (40, 40)], [(513, 64), (1025, 33)], [(3080, 33)],
            [(4100, 34), (100, 3)]]


@pytest.mark.parametrize("dt,shapes", [(np.float32, s) for s in SHAPES32] + [(np.float64, s) for s in SHAPES64])
def test_blocked_qr_edges(dt, shapes):
    import paper_1707_05141_gb300 as bs
    bs.build()
    rng = np.random.default_rng(5)
    mats = [rng.standard_normal(s).astype(dt) for s in shapes]
    m, n = (np.array([s[i] for s in shapes], np.int32) for i in (0, 1))
    for pad in (0, 3):   # aligned where the rows are, and odd leading dimensions on an odd element
        ld = m + pad
        off = np.concatenate([[0], np.cumsum((ld * n.astype(np.int64) + 3) // 4 * 4)]) + (1 if pad else 0)
        flat = np.full(int(off[-1]) + 8, 3.0, dt)
        for a, o, l in zip(mats, off, ld):
            for j in range(a.shape[1]):
                flat[o + j * l:o + j * l + a.shape[0]] = a[:, j]
        t = torch.from_numpy(flat).cuda()
        q, r = torch.zeros_like(t), torch.zeros(int((n.astype(np.int64) ** 2 + 3).sum()), dtype=t.dtype, device="cuda")
        ro = np.concatenate([[0], np.cumsum(n.astype(np.int64) ** 2)])
        A, Q, R = bs.Batch.packed(t, off[:-1], m, n, ld), bs.Batch.packed(q, off[:-1], m, n, ld), bs.Batch.packed(r, ro[:-1], n, n, n)
        info = torch.full((len(m),), 7, dtype=torch.int32, device="cuda")
        ws = torch.empty(bs.batched_qr_blocked_workspace(A), dtype=torch.uint8, device="cuda")
        bs.batched_qr_blocked(A, Q, R, info, ws)
        torch.cuda.synchronize()
        assert (info.cpu().numpy() == 0).all()
        qh, rh = q.cpu().numpy().astype(np.float64), r.cpu().numpy().astype(np.float64)
        for b, a in enumerate(mats):
            a = a.astype(np.float64)
            mm, nn = a.shape
            Qb = np.stack([qh[off[b] + j * ld[b]:][:mm] for j in range(nn)], 1)
            Rb = rh[ro[b]:ro[b] + nn * nn].reshape(nn, nn).T
            assert np.array_equal(np.tril(Rb, -1), np.zeros((nn, nn)))
            assert np.abs(Qb.T @ Qb - np.eye(nn)).max() <= gate(dt), a.shape
            assert np.linalg.norm(a - Qb @ Rb) <= gate(dt) * np.linalg.norm(a), a.shape
            ref = np.linalg.qr(a, mode="r")   # the reflectors' signs are LAPACK's, but for a square's last row
            if mm == nn:
                ref[-1] *= -1
            assert np.abs(Rb - ref).max() <= 64 * np.finfo(dt).eps * np.sqrt(mm) * np.linalg.norm(a, 2), a.shape
