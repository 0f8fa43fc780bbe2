"""The work a user of this library has it do, as measurable cases.

A case names one call through the public entry points with its sizes, element type and options;
``prepare`` makes what the caller has in hand before the call, ``run`` makes the call, ``exact`` says
what the call's numbers are in 64-bit arithmetic.  Sizes are the library's own workloads, sizes of its
tests, or generic ones; ``draw`` spreads over the ranges that the listed cases stand for.
"""
from __future__ import annotations

import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_1707_05141_gb300 as bs

POOL = 16   # Haar factors per side that a batch's matrices draw from


def listed():
    return [
        # one front of a tree code compresses a handful of small blocks: latency and launches count
        dict(name="svd_few_33x20", kind="svd", dtype="f32", batch=16, m=33, n=20, spectrum="exp8", call="plain",
             tuned=False, vectors=True),
        # the headline batch: small square blocks of a hierarchical matrix, register tier, tuned variant
        dict(name="svd_64x64", kind="svd", dtype="f32", batch=20000, m=64, n=64, spectrum="exp8", call="plan",
             tuned=True, vectors=True),
        # double precision, condition number 1e8
        dict(name="svd_f64_32x32", kind="svd", dtype="f64", batch=1000, m=32, n=32, spectrum="graded8", call="plan",
             tuned=True, vectors=True),
        # blocks beyond the register tier, odd sizes
        dict(name="svd_127x100", kind="svd", dtype="f32", batch=1000, m=127, n=100, spectrum="exp8", call="plan",
             tuned=False, vectors=True),
        # the headline QR batch: narrow panels
        dict(name="qr_128x32", kind="qr", dtype="f32", batch=20000, m=128, n=32, spectrum="exp8", call="plan"),
        # tall sample panels of a randomized SVD, odd sizes
        dict(name="qr_250x149", kind="qr", dtype="f32", batch=2000, m=250, n=149, spectrum="gauss", call="plan"),
        # blocked QR of matrices that live in global memory
        dict(name="qr_blocked_2000x600", kind="qr_blocked", dtype="f32", batch=8, m=2000, n=600, spectrum="gauss",
             call="plan"),
        # the block-Jacobi workload: large squares, spectrum over six decades, QR-preconditioned, tuned inner variant
        dict(name="block_512x512", kind="block", dtype="f32", batch=500, m=512, n=512, spectrum="loguniform",
             call="plan", precondition=True, tuned=True),
        # a user's plain call on two middle-sized matrices
        dict(name="block_few_300x200", kind="block", dtype="f32", batch=2, m=300, n=200, spectrum="exp8",
             call="plain", precondition=False, tuned=False),
        # compression of uneven blocks to a tolerance with rank guesses
        dict(name="rsvd_uneven", kind="rsvd", dtype="f32", batch=16384, lo=64, hi=256, shapes="pow2", mode="tol",
             tol=1e-5, hints=True, rank=0, sizes=1),
        # truncation of a nested basis, level by level
        dict(name="h2_depth12", kind="h2", dtype="f32", depth=12, q=8, eps=1e-5),
        # one training step of the rank predictor
        dict(name="rank_train", kind="train", batch=2048),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svd", "svd", "svd", "qr", "qr", "qr_blocked", "block", "block", "rsvd", "rsvd", "h2", "train"])
    if kind == "svd":
        dtype = rng.choice(["f32", "f32", "f64"])
        n = _log_int(rng, 4, 128 if dtype == "f32" else 64)
        m = min(_log_int(rng, n, 2 * n + 8), 128 if dtype == "f32" else 64)
        if rng.random() < 0.3:
            m, n = n, m
        work = m * n * min(m, n)
        batch = max(1, min(_log_int(rng, 4, 20000), int((2.5e9 if dtype == "f32" else 6e7) / work)))
        return dict(kind="svd", dtype=dtype, batch=batch, m=m, n=n,
                    spectrum=rng.choice(["exp8", "loguniform", "gauss"]) if dtype == "f32" else "graded8",
                    call="plain" if batch <= 64 else "plan", tuned=m == n and 16 < n <= 64 and rng.random() < 0.6,
                    vectors=rng.random() < 0.8)
    if kind == "qr":
        dtype = rng.choice(["f32", "f32", "f64"])
        n = _log_int(rng, 4, 160 if dtype == "f32" else 96)
        # Q is determined to the precision of the input only up to the condition number: squares and wide
        # spectra stay narrow, Gaussian panels stay tall
        exp8 = n <= 48 and rng.random() < 0.5
        m = min(_log_int(rng, n if exp8 else 5 * n // 4 + 8, 4 * n + 16), 300)
        batch = max(1, min(_log_int(rng, 4, 20000), int((8e8 if dtype == "f32" else 1.5e8) / (m * n * math.sqrt(n)))))
        return dict(kind="qr", dtype=dtype, batch=batch, m=m, n=n, spectrum="exp8" if exp8 else "gauss",
                    call="plain" if batch <= 64 else "plan")
    if kind == "qr_blocked":
        dtype = rng.choice(["f32", "f32", "f64"])
        m = _log_int(rng, 200, 5000)
        n = min(4 * m // 5 - 8, _log_int(rng, 33, 700))
        batch = max(1, min(_log_int(rng, 1, 64), int((1.2e10 if dtype == "f32" else 8e8) / (m * n * n))))
        return dict(kind="qr_blocked", dtype=dtype, batch=batch, m=m, n=n, spectrum="gauss",
                    call=rng.choice(["plain", "plan"]))
    if kind == "block":
        n = _log_int(rng, 70, 512)
        m = min(_log_int(rng, n, 2 * n), 700)
        if rng.random() < 0.3:
            m, n = n, m
        batch = max(1, min(_log_int(rng, 1, 300), int(3e10 / (m * n * min(m, n)))))
        pre = rng.random() < 0.6
        return dict(kind="block", dtype="f32", batch=batch, m=m, n=n, spectrum=rng.choice(["exp8", "loguniform"]),
                    call="plain" if batch <= 8 else "plan", precondition=pre, tuned=rng.random() < 0.5)
    if kind == "rsvd":
        hi = rng.choice([64, 128, 200, 256])
        batch = _log_int(rng, 16, 8192)
        mode = rng.choice(["tol", "tol", "rank"])
        return dict(kind="rsvd", dtype="f32", batch=batch, lo=min(64, hi // 2), hi=hi,
                    shapes=rng.choice(["pow2", "any"]), mode=mode, tol=rng.choice([1e-3, 1e-5]),
                    hints=rng.random() < 0.6, rank=rng.randrange(5, 25) if mode == "rank" else 0, sizes=rng.randrange(1000))
    if kind == "h2":
        return dict(kind="h2", dtype=rng.choice(["f32", "f32", "f64"]), depth=rng.randrange(4, 10), q=rng.randrange(3, 9),
                    eps=rng.choice([1e-3, 1e-5]))
    return dict(kind="train", batch=_log_int(rng, 64, 16384))


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------

def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 17)
    return g


def _haar(count, rows, cols, g):
    """``count`` Haar-distributed rows x cols orthonormal factors in 64 bits."""
    q, r = torch.linalg.qr(torch.randn((count, rows, cols), generator=g, device="cuda", dtype=torch.float64))
    return q * torch.where(torch.diagonal(r, dim1=-2, dim2=-1) < 0, -1.0, 1.0)[:, None, :]


def _sigma(spectrum, batch, k, g):
    i = torch.arange(k, device="cuda", dtype=torch.float64)
    if spectrum == "exp8":
        s = torch.exp(-i / 8).expand(batch, k)
    elif spectrum == "graded8":
        s = (10.0 ** (-8.0 * i / max(k - 1, 1))).expand(batch, k)
    else:   # log-uniform on [1e-6, 1]
        u = torch.rand((batch, k), generator=g, device="cuda", dtype=torch.float64)
        s = torch.exp(math.log(1e-6) * (1 - u)).sort(dim=1, descending=True).values
    return s


def _matrices(batch, m, n, s, g, pools=None):
    """U diag(s) V^T with random signs on Haar factors from a pool, stored column by column: (batch, n, m)."""
    k = min(m, n)
    pu, pv = pools if pools else (_haar(min(POOL, batch), m, k, g), _haar(min(POOL, batch), n, k, g))
    out = torch.empty((batch, n, m), device="cuda", dtype=torch.float64)
    step = max(1, int(1e8) // (m * n))
    for b0 in range(0, batch, step):
        c = min(step, batch - b0)
        iu = torch.randint(0, pu.shape[0], (c,), generator=g, device="cuda")
        iv = torch.randint(0, pv.shape[0], (c,), generator=g, device="cuda")
        sm = torch.randint(0, 2, (c, 1, m), generator=g, device="cuda").double() * 2 - 1
        sn = torch.randint(0, 2, (c, n, 1), generator=g, device="cuda").double() * 2 - 1
        pick = lambda p, i: p[i][:, :, :k]  # noqa: E731
        v = pick(pv, iv) * s[b0:b0 + c, None, :]
        out[b0:b0 + c] = torch.bmm(v, pick(pu, iu).transpose(1, 2)) * sm * sn
    return out


def _uniform_input(case, seed):
    g = _gen(seed)
    b, m, n = case["batch"], case["m"], case["n"]
    if case["spectrum"] == "gauss":
        return torch.randn((b, n, m), generator=g, device="cuda", dtype=torch.float64).to(_dtype(case))
    return _matrices(b, m, n, _sigma(case["spectrum"], b, min(m, n), g), g).to(_dtype(case))


def _uneven_sizes(case):
    rng = np.random.default_rng([case["sizes"], 3])
    b, lo, hi = case["batch"], case["lo"], case["hi"]
    if case["shapes"] == "pow2":
        choices = np.array([x for x in (64, 128, 256) if lo <= x <= hi], np.int32)
        m, n = rng.choice(choices, b), rng.choice(choices, b)
    else:   # a few odd shapes
        choices = rng.integers(lo, hi + 1, 6).astype(np.int32)
        m, n = rng.choice(choices, b), rng.choice(choices, b)
    return m.astype(np.int32), n.astype(np.int32), rng.uniform(2.0, 12.0, b)


def _uneven_input(case, seed):
    """Blocks packed in one tensor, sigma_i = exp(-i / r0) with r0 uniform on [2, 12]."""
    g = _gen(seed)
    m, n, r0 = _uneven_sizes(case)
    size = (m.astype(np.int64) * n + 3) // 4 * 4
    off = np.concatenate([[0], np.cumsum(size)[:-1]]).astype(np.int64)
    flat = torch.zeros(int(size.sum()), device="cuda", dtype=_dtype(case))
    dims = sorted(set(m.tolist()) | set(n.tolist()))
    pool = {d: _haar(POOL, d, d, g) for d in dims}
    for mm in dims:
        for nn in dims:
            sel = np.nonzero((m == mm) & (n == nn))[0]
            if len(sel) == 0:
                continue
            k = min(mm, nn)
            s = torch.exp(-torch.arange(k, device="cuda", dtype=torch.float64)[None, :]
                          / torch.as_tensor(r0[sel], device="cuda")[:, None])
            a = _matrices(len(sel), mm, nn, s, g, (pool[mm], pool[nn])).to(flat.dtype).reshape(len(sel), -1)
            pos = torch.as_tensor(off[sel], device="cuda")[:, None] + torch.arange(mm * nn, device="cuda")
            flat[pos.reshape(-1)] = a.reshape(-1)
    return flat, off, m, n, r0


def _lagrange(lo, hi, q, x):
    """Lagrange polynomials on the q Chebyshev points of [lo, hi] at x: (..., q)."""
    j = np.arange(q)
    nodes = 0.5 * (lo + hi)[..., None] + 0.5 * (hi - lo)[..., None] * np.cos((2.0 * j + 1.0) * math.pi / (2.0 * q))
    out = np.ones(x.shape + (q,))
    for a in range(q):
        for b in range(q):
            if b != a:
                out[..., a] *= (x - nodes[..., b]) / (nodes[..., a] - nodes[..., b])
    return out, nodes


def _basis_tree(depth, q, seed):
    """Chebyshev-interpolation row basis of a k-d tree over a perturbed grid of the unit square, about 64
    points a leaf; each box is cut across its longer side within a point of the median, the same
    counts for every seed."""
    rng, shape = np.random.default_rng([int(seed), 5]), np.random.default_rng([depth, 7])
    side = int(round(math.sqrt(64 * 2 ** depth)))
    i, j = np.meshgrid(np.arange(side), np.arange(side), indexing="ij")
    pts = (np.stack([i.ravel(), j.ravel()], 1) + 0.5 + rng.uniform(-0.45, 0.45, (side * side, 2))) / side
    count, lo, hi = np.array([len(pts)]), [np.zeros((1, 2))], [np.ones((1, 2))]
    node = np.zeros(len(pts), np.int64)
    for l in range(depth):
        r = np.arange(1 << l)
        d = np.argmax(hi[l] - lo[l], axis=1)
        x = pts[np.arange(len(pts)), d[node]]
        order = np.lexsort((x, node))
        pts, node, x = pts[order], node[order], x[order]
        left = count // 2 + shape.integers(-1, 2, len(count))
        first = np.cumsum(count) - count
        cut = 0.5 * (x[first + left - 1] + x[first + left])
        node = 2 * node + (np.arange(len(pts)) - first[node] >= left[node])
        count = np.stack([left, count - left], 1).ravel()
        lo2, hi2 = np.repeat(lo[l], 2, 0), np.repeat(hi[l], 2, 0)
        hi2[2 * r, d], lo2[2 * r + 1, d] = cut, cut
        lo.append(lo2)
        hi.append(hi2)
    lx, _ = _lagrange(lo[depth][node, 0], hi[depth][node, 0], q, pts[:, 0])
    ly, _ = _lagrange(lo[depth][node, 1], hi[depth][node, 1], q, pts[:, 1])
    rows = (lx[:, :, None] * ly[:, None, :]).reshape(len(pts), q * q)
    leaves = np.split(rows, np.cumsum(count)[:-1])
    transfers = [[]]
    for l in range(1, depth + 1):
        parent = np.arange(1 << l) // 2
        one = []
        for d in (0, 1):
            _, xi = _lagrange(lo[l][:, d], hi[l][:, d], q, lo[l][:, d])
            one.append(_lagrange(lo[l - 1][parent, None, d], hi[l - 1][parent, None, d], q, xi)[0])
        e = one[0][:, :, None, :, None] * one[1][:, None, :, None, :]
        transfers.append(list(e.reshape(1 << l, q * q, q * q)))
    return leaves, transfers


def _train_input(case, seed):
    g = _gen(seed)
    randn = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float32)  # noqa: E731
    h, f, b = 64, bs.SKETCH_FEATURES, case["batch"]
    params = torch.cat([randn(h * f) * math.sqrt(2 / f), randn(h) * 0.1, randn(h * h) * math.sqrt(2 / h),
                        randn(h) * 0.1, randn(h) * math.sqrt(1 / h), torch.ones(1, device="cuda")])
    rank = torch.randint(1, 130, (b,), generator=g, device="cuda")
    # moments as in the middle of a training run
    mom, vel = randn(params.numel()) * 1e-2, (1 + randn(params.numel()).abs()) * 1e-3
    return dict(x=randn(b, f), target=torch.log(rank.float() + 1), params=params, mom=mom, vel=vel)


# ----------------------------------------------------------------------------------------------
# what the caller has in hand, and the call
# ----------------------------------------------------------------------------------------------

def _tuned_variant(code, m, n, precondition):
    """The register variant the autotuner records on this GPU for square blocks: carried column norms,
    QR-preconditioned (plain for the block tier's inner SVDs)."""
    for k in range(1, bs.jacobi_variants(code, m, n, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(code, m, n, k)
        if d["carried_norms"] and bool(d["qr_precond"]) == precondition:
            return k
    return 0


def _empty(shape, dtype):
    return torch.zeros(shape, device="cuda", dtype=dtype)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        s = _train_input(case, seed)
        s.update(grad=torch.zeros_like(s["params"]), loss=_empty(1, torch.float32), step=100)
        return dict(case=case, **s)
    if kind == "h2":
        leaves, transfers = _basis_tree(case["depth"], case["q"], seed)
        return dict(case=case, plan=bs.H2Plan(leaves, transfers, case["q"] ** 2, _dtype(case)))
    if kind == "rsvd":
        flat, off, m, n, r0 = _uneven_input(case, seed)
        k = np.minimum(m, n)
        pack = lambda cnt: np.concatenate([[0], np.cumsum((cnt + 3) // 4 * 4)]).astype(np.int64)  # noqa: E731
        ou, ov, os_ = pack(m.astype(np.int64) * k), pack(n.astype(np.int64) * k), pack(k.astype(np.int64))
        dt = flat.dtype
        u, v, s = _empty(int(ou[-1]), dt), _empty(int(ov[-1]), dt), _empty(int(os_[-1]), dt)
        A = bs.Batch.packed(flat, off, m, n)
        ints = lambda x: torch.as_tensor(np.asarray(x, np.int32), device="cuda")  # noqa: E731
        hint = np.minimum(np.ceil(r0 * math.log(1 / case["tol"])), k)
        b = case["batch"]
        return dict(case=case, A=A, U=bs.Batch.packed(u, ou[:-1], m, k), V=bs.Batch.packed(v, ov[:-1], n, k),
                    S=bs.Batch.packed(s, os_[:-1], k, np.ones_like(k)), kmax=ints(k), u=u, v=v, s=s,
                    rank=_empty(b, torch.int32), info=_empty(b, torch.int32), samples=_empty(b, torch.int32),
                    err=_empty(b, torch.float32), hint=ints(hint) if case["hints"] else None,
                    fixed=ints(np.full(b, case["rank"])) if case["mode"] == "rank" else None,
                    ws=torch.empty(bs.batched_rsvd_workspace(A, m, n), dtype=torch.uint8, device="cuda"))
    a = _uniform_input(case, seed)
    st = dict(case=case, a=a)
    if kind == "svd":
        st["tier"] = bs.TIER_AUTO
        if case["tuned"]:
            code = bs.F32 if a.dtype == torch.float32 else bs.F64
            k = _tuned_variant(code, case["m"], case["n"], True)
            st["tier"] = bs.TIER_REGISTER | (k << 8) if k else bs.TIER_AUTO
    if kind == "block":
        k = _tuned_variant(bs.F32, 64, 64, False) if case["tuned"] else 0
        st["method"] = bs.BLOCK_GRAM | (bs.BLOCK_QR_PRECONDITION if case["precondition"] else 0) | (k << 8)
    if case["call"] == "plain":
        return st
    b, m, n, dt = case["batch"], case["m"], case["n"], a.dtype
    k = min(m, n)
    st["A"], st["info"] = bs.Batch.uniform(a, m, n), _empty(b, torch.int32)
    if kind in ("qr", "qr_blocked"):
        st["q"], st["r"] = _empty((b, n, m), dt), _empty((b, n, n), dt)
        st["Q"], st["R"] = bs.Batch.uniform(st["q"], m, n), bs.Batch.uniform(st["r"], n, n)
        if kind == "qr_blocked":
            st["ws"] = torch.empty(bs.batched_qr_blocked_workspace(st["A"]), dtype=torch.uint8, device="cuda")
        return st
    st["s"] = _empty((b, 1, k), dt)
    st["S"] = bs.Batch.uniform(st["s"], k, 1)
    st["U"] = st["V"] = st["u"] = st["v"] = None
    if case.get("vectors", True):
        st["u"], st["v"] = _empty((b, k, m), dt), _empty((b, k, n), dt)
        st["U"], st["V"] = bs.Batch.uniform(st["u"], m, k), bs.Batch.uniform(st["v"], n, k)
    if kind == "block":
        size = bs.batched_svd_block_jacobi_workspace(st["A"], 32, st["method"])
        st["ws"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    return st


def run(state):
    st, case = state, state["case"]
    kind = case["kind"]
    if kind == "train":
        bs.bsvd_mlp_grad(st["x"], st["target"], st["params"], st["grad"], st["loss"])
        bs.bsvd_mlp_adam(st["params"], st["grad"], st["mom"], st["vel"], st["step"])
        return {k: st[k] for k in ("grad", "loss", "params", "mom", "vel")}
    if kind == "h2":
        p = st["plan"]
        p.run(case["eps"])
        return dict(new_leaf=p.new_leaf, new_transfer=p.new_transfer, T=p.T, rank=p.rank, info=p.info,
                    rotations=p.rotations)
    if kind == "rsvd":
        bs.batched_rsvd(st["A"], st["U"], st["S"], st["V"], st["kmax"], st["rank"], st["info"], st["ws"], st["hint"],
                        tol=case["tol"], seed=1707, err_est=st["err"], samples=st["samples"], fixed_rank=st["fixed"])
        return {k: st[k] for k in ("u", "s", "v", "rank", "info", "err", "samples")}
    if kind == "svd":
        if case["call"] == "plain":
            u, s, v, info, rotations = bs.svd(st["a"], case["vectors"], case["vectors"], tier=st["tier"])
            return dict(u=u, s=s, v=v, info=info, rotations=rotations)
        bs.batched_svd_jacobi(st["A"], st["S"], st["U"], st["V"], st["info"], tier=st["tier"])
        return dict(u=st["u"], s=st["s"], v=st["v"], info=st["info"])
    if kind == "block":
        if case["call"] == "plain":
            u, s, v, info, rotations = bs.svd_block(st["a"], method=st["method"])
            return dict(u=u, s=s, v=v, info=info, rotations=rotations)
        bs.batched_svd_block_jacobi(st["A"], st["S"], st["U"], st["V"], st["info"], st["ws"], method=st["method"])
        return dict(u=st["u"], s=st["s"], v=st["v"], info=st["info"])
    if case["call"] == "plain":
        q, r, info = (bs.qr if kind == "qr" else bs.qr_blocked)(st["a"])
        return dict(q=q, r=r, info=info)
    if kind == "qr":
        bs.batched_qr(st["A"], st["Q"], st["R"], st["info"])
    else:
        bs.batched_qr_blocked(st["A"], st["Q"], st["R"], st["info"], st["ws"])
    return dict(q=st["q"], r=st["r"], info=st["info"])


# ----------------------------------------------------------------------------------------------
# what a pass cannot do without, and what its numbers are
# ----------------------------------------------------------------------------------------------

def _svd_flops(m, n):
    m, n = max(m, n), min(m, n)
    return 14.0 * m * n * n + 8.0 * n ** 3   # reduced factorisation with both sets of vectors


def work(case):
    kind = case["kind"]
    if kind == "train":
        p = bs.MLP_PARAMS
        return dict(bytes=4.0 * (case["batch"] * (bs.SKETCH_FEATURES + 1) + 7 * p), flops=6.0 * case["batch"] * p)
    es = 4 if case["dtype"] == "f32" else 8
    if kind == "h2":
        k, leaves = case["q"] ** 2, 1 << case["depth"]
        rows = 64.0 * leaves
        elems = 2 * rows * k + leaves * 2 * (2.0 * k * k) + leaves * 2.0 * k * k
        return dict(bytes=es * elems, flops=leaves * _svd_flops(64, k) + leaves * (_svd_flops(2 * k, k) + 4.0 * k ** 3))
    if kind == "rsvd":
        m, n, r0 = (x.astype(np.float64) for x in _uneven_sizes(case))
        k = np.minimum(m, n)
        r = np.full(len(m), float(case["rank"])) if case["mode"] == "rank" else np.minimum(
            np.ceil(r0 * math.log(1 / case["tol"])), k)
        l = np.minimum(r + 8, k)
        return dict(bytes=es * float((m * n + (m + n + 1) * r).sum()),
                    flops=float((8 * m * n * l + 6 * (m + n) * l * l + 22 * l ** 3).sum()))
    b, m, n = case["batch"], case["m"], case["n"]
    k = min(m, n)
    if kind in ("svd", "block"):
        vec = case.get("vectors", True)
        return dict(bytes=float(es * b) * (m * n + k + (k * (m + n) if vec else 0)),
                    flops=b * (_svd_flops(m, n) if vec else 4.0 * max(m, n) * k * k - 4.0 * k ** 3 / 3))
    return dict(bytes=float(es * b) * (2 * m * n + n * n), flops=b * (4.0 * m * n * n - 4.0 * n ** 3 / 3))


def _over_batch(fn, a):
    """fn over chunks of the batch ``a`` on the host's cores."""
    parts = np.array_split(a, max(1, min(len(a), 64)))
    with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
        return list(ex.map(fn, parts))


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind not in ("svd", "block", "qr", "qr_blocked"):
        return None   # singular vectors to a tolerance: no value of their own beyond signs and truncation
    a = _uniform_input(case, seed).transpose(1, 2).double().cpu().numpy()
    if kind in ("svd", "block"):
        if kind == "block" and case["batch"] * case["m"] * case["n"] * min(case["m"], case["n"]) > 3e10:
            return None   # minutes of LAPACK
        s = torch.from_numpy(np.concatenate(_over_batch(lambda x: np.linalg.svd(x, compute_uv=False), a)))
        if case["call"] == "plan":
            s = s[:, None, :]
        return dict(u=None, s=s, v=None, info=None)   # singular vectors: signs are the method's
    parts = _over_batch(np.linalg.qr, a)
    q, r = (np.concatenate([p[i] for p in parts]) for i in (0, 1))
    if case["m"] == case["n"]:   # LAPACK leaves the last entry of a square matrix, Algorithm 1 reflects it
        q[:, :, -1] *= -1
        r[:, -1, :] *= -1
    return dict(q=torch.from_numpy(np.ascontiguousarray(q.transpose(0, 2, 1))),
                r=torch.from_numpy(np.ascontiguousarray(r.transpose(0, 2, 1))), info=None)


def _exact_train(case, seed):
    t = {k: v.double() for k, v in _train_input(case, seed).items()}
    h, f, b, step = 64, bs.SKETCH_FEATURES, case["batch"], 100
    p = t["params"].clone().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [h * f, h, h * h, h, h, 1])
    y = torch.relu(torch.relu(t["x"] @ w1.view(h, f).T + b1) @ w2.view(h, h).T + b2) @ w3 + b3
    loss = ((y - t["target"]) ** 2).sum() / (2 * b)
    (grad,) = torch.autograd.grad(loss, p)
    mom, vel = 0.9 * t["mom"] + 0.1 * grad, 0.999 * t["vel"] + 0.001 * grad ** 2
    new = t["params"] - 1e-3 * (mom / (1 - 0.9 ** step)) / (torch.sqrt(vel / (1 - 0.999 ** step)) + 1e-8)
    return dict(grad=grad, loss=loss.detach().reshape(1), params=new, mom=mom, vel=vel)
