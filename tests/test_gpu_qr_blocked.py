"""GPU parity of the QRs with panels in registers: copies in the workspace and Q of different alignment, columns
across the type's range, more matrices than SMs."""
import numpy as np
import pytest

from parity import gate

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run_qr(mats, ldq=None, blocked=True):
    """Q, R (64 bits) and info of a batch of matrices of one type; column j of Q starts on a multiple of ldq[b]
    elements after a 16-byte boundary."""
    import paper_1707_05141_gb300 as bs
    bs.build()
    m, n = (np.array([a.shape[i] for a in mats], np.int32) for i in (0, 1))
    ldq = m if ldq is None else np.asarray(ldq, np.int32)

    def pack(ld, cols):
        off = np.concatenate([[0], np.cumsum((ld.astype(np.int64) * np.maximum(cols, 1) + 3) // 4 * 4)])
        return np.zeros(int(off[-1]) + 4, mats[0].dtype), off[:-1]

    (fa, oa), (fq, oq), (fr, orr) = pack(m, n), pack(ldq, n), pack(n, n)
    for a, o in zip(mats, oa):
        fa[o:o + a.size] = a.T.reshape(-1)
    ta, tq, tr = (torch.from_numpy(x).cuda() for x in (fa, fq, fr))
    A, Q, R = bs.Batch.packed(ta, oa, m, n), bs.Batch.packed(tq, oq, m, n, ldq), bs.Batch.packed(tr, orr, n, n)
    info = torch.full((len(mats),), 7, dtype=torch.int32, device="cuda")
    if blocked:
        ws = torch.empty(bs.batched_qr_blocked_workspace(A), dtype=torch.uint8, device="cuda")
        bs.batched_qr_blocked(A, Q, R, info, ws)
    else:
        bs.batched_qr(A, Q, R, info)
    torch.cuda.synchronize()
    hq, hr = tq.cpu().numpy().astype(np.float64), tr.cpu().numpy().astype(np.float64)
    q = [np.stack([hq[o + j * l:][:mm] for j in range(nn)], 1) for o, l, mm, nn in zip(oq, ldq, m, n)]
    r = [hr[o:o + nn * nn].reshape(nn, nn).T for o, nn in zip(orr, n)]
    return q, r, info.cpu().numpy()


# (the workspace holds matrix b at b max_m max_n elements: misaligned for an odd product and an odd b, while
# Q's columns are 16-byte aligned, so V and C of a block reflector are copied by different means)
@pytest.mark.parametrize("dt,shapes", [(np.float32, [(257, 65), (256, 64), (256, 33), (252, 65)]),
                                       (np.float32, [(2001, 601), (2001, 601)]),
                                       (np.float32, [(33, 33), (32, 1), (29, 29)]),
                                       (np.float64, [(131, 33), (128, 33), (130, 1)])])
def test_aligned_q_beside_unaligned_workspace(dt, shapes):
    rng = np.random.default_rng(2)
    mats = [rng.standard_normal(s).astype(dt) for s in shapes]
    assert max(s[0] for s in shapes) * max(s[1] for s in shapes) % 2 == 1
    q, r, info = run_qr(mats, [(s[0] + 3) // 4 * 4 for s in shapes])
    assert (info == 0).all()
    for a, qq, rr in zip(mats, q, r):
        a = a.astype(np.float64)
        assert np.abs(qq.T @ qq - np.eye(a.shape[1])).max() <= gate(dt), a.shape
        assert np.linalg.norm(a - qq @ rr) <= gate(dt) * np.linalg.norm(a), a.shape
        assert not np.tril(rr, -1).any()


# the blocked one-CTA QR, and the blocked QR with one CTA, a cluster of two and one of four per panel
@pytest.mark.parametrize("dt,m,n,blocked", [(np.float32, 200, 80, False), (np.float32, 300, 66, False),
                                            (np.float32, 200, 80, True), (np.float32, 600, 40, True),
                                            (np.float32, 2000, 64, True), (np.float64, 200, 40, True),
                                            (np.float64, 1100, 33, True)])
def test_columns_across_the_range(dt, m, n, blocked):
    """Norms in the type's range are enough, also where the product of two columns' norms is not; dependent columns
    (whose remainder after the first reflector is rounding) and independent ones."""
    rng = np.random.default_rng(4)
    a = rng.standard_normal((m, n))
    big, small = (1e17, 1e-17) if dt == np.float32 else (1e150, 1e-150)
    far = 1e5 if dt == np.float32 else 1e50
    mats = []
    for head, factor in ((big, far), (small, 1 / far)):
        x = a.copy()
        x[:, 0] *= head
        x[:, 3] = x[:, 0] * factor   # a multiple of column 0
        x[:, n - 1] = x[:, 0] / factor
        mats.append(x.astype(dt))
    mats += [(a * big).astype(dt), (a * small).astype(dt), (a * (small / 1e3)).astype(dt)]
    x = a.copy()
    x[:, 5] *= big
    x[:, n - 2] *= small
    mats.append(x.astype(dt))
    q, r, info = run_qr(mats, blocked=blocked)
    assert (info == 0).all()
    for i, (x, qq, rr) in enumerate(zip(mats, q, r)):
        x = x.astype(np.longdouble)
        assert np.abs(qq.T @ qq - np.eye(n)).max() <= gate(dt), i
        size = np.sqrt((x * x).sum(0))
        assert (np.sqrt(((qq.astype(np.longdouble) @ rr.astype(np.longdouble) - x) ** 2).sum(0)) <= gate(dt) * size).all(), i


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("m", [100, 2000])
def test_nan_stays_in_r(dt, m):
    """No entry of R that a NaN reaches is a number, the diagonal included."""
    rng = np.random.default_rng(6)
    mats = [rng.standard_normal((m, n)).astype(dt) for n in (33, 1, 40)]
    mats[0][m // 2, 32] = np.nan
    mats[1][0, 0] = np.nan
    mats[2][m - 1, 7] = np.nan
    _, r, _ = run_qr(mats)
    assert np.isnan(r[0][:, 32]).all() and np.isfinite(r[0][:, :32]).all()
    assert np.isnan(r[1]).all()
    assert np.isnan(r[2][:8, 7]).all()
    assert np.isnan(np.diag(r[2])[7:]).all() and np.isfinite(r[2][:, :7]).all()


# more matrices than SMs take the panels with half of the registers a thread; 32, 64, 128 and 256 rows are their sizes
@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("rows", [[33, 40, 64], [65, 66, 128], [129, 200, 256], [257, 300, 288]])
def test_more_matrices_than_sms(dt, rows):
    rng = np.random.default_rng(rows[0])
    shapes = [(rows[i % 3], n) for i, n in enumerate(rng.integers(1, 38, 165))]
    mats = [rng.standard_normal((m, min(m, n))).astype(dt) for m, n in shapes]
    mats[7][:, 0] = 0
    q, r, info = run_qr(mats)
    assert (info == 0).all()
    for b, (a, qq, rr) in enumerate(zip(mats, q, r)):
        a = a.astype(np.float64)
        assert np.abs(qq.T @ qq - np.eye(a.shape[1])).max() <= gate(dt), (b, a.shape)
        assert np.linalg.norm(a - qq @ rr) <= gate(dt) * np.linalg.norm(a), (b, a.shape)
        assert not np.tril(rr, -1).any()
