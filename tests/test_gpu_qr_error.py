"""The blocked one-CTA QR (FP32) errs no more against 64 bits than Algorithm 1 applied one reflector at a time, whose
FP32 arithmetic (sums over 32 lanes and a tree) is carried out here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F32, F64 = np.float32, np.float64


def _fma(a, b, c):
    return (a.astype(F64) * b.astype(F64) + c.astype(F64)).astype(F32)


def _dot(v, x):
    """v^T x: row r in lane r mod 32, a chain of FMAs per lane, then the butterfly."""
    t = -(-len(v) // 32)
    v = np.concatenate([v, np.zeros(32 * t - len(v), F32)]).reshape(t, 32, 1)
    x = np.concatenate([x, np.zeros((32 * t - len(x), x.shape[1]), F32)]).reshape(t, 32, -1)
    s = np.zeros(x.shape[1:], F32)
    for k in range(t):
        s = _fma(v[k], x[k], s)
    while len(s) > 1:
        s = s[:len(s) // 2] + s[len(s) // 2:]
    return s[0]


def one_reflector_at_a_time(a):
    m, n = a.shape
    a, diag, vs = a.copy(), np.zeros(n, F32), []
    for i in range(n):
        x = a[i:, i].copy()
        alpha = np.sqrt(_dot(x, x[:, None])[0])
        inv = F32(1 / np.sqrt(F64(F32(2) * alpha * (alpha + abs(x[0])))))
        diag[i] = -alpha if x[0] >= 0 else alpha
        x[0] -= diag[i]
        vs.append(x * inv)
        w = F32(-2) * _dot(vs[i], a[i:, i + 1:]) if i + 1 < n else np.zeros(0, F32)
        a[i:, i + 1:] = _fma(w[None, :], vs[i][:, None], a[i:, i + 1:])
    q = np.eye(m, n, dtype=F32)
    for i in range(n - 1, -1, -1):
        w = F32(-2) * _dot(vs[i], q[i:, i:])
        q[i:, i:] = _fma(w[None, :], vs[i][:, None], q[i:, i:])
    return q, np.triu(a[:n], 1) + np.diag(diag)


@pytest.mark.parametrize("m,n", [(250, 149), (160, 120), (200, 80), (300, 66), (140, 66), (257, 64), (300, 50)])
def test_error_against_64_bits(m, n):
    import paper_1707_05141_gb300 as bs
    bs.build()
    b = 6
    a = np.random.default_rng(m + n).standard_normal((b, m, n)).astype(F32)
    q, r, info = bs.qr(torch.from_numpy(np.ascontiguousarray(a.transpose(0, 2, 1))).cuda())
    assert info.tolist() == [0] * b
    q, r = (x.cpu().numpy().transpose(0, 2, 1).astype(F64) for x in (q, r))
    qe, re = np.linalg.qr(a.astype(F64))
    ref = [one_reflector_at_a_time(x) for x in a]
    for got, exact, one in ((q, qe, [x[0] for x in ref]), (r, re, [x[1] for x in ref])):
        assert np.linalg.norm(got - exact) <= np.linalg.norm(np.stack(one).astype(F64) - exact)
