"""A null entry in the pointer array of U or V leaves that matrix's factor unwritten and the others as they are."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _variant(bs, m, n, **want):
    for k in range(1, bs.jacobi_variants(bs.F32, m, n, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(bs.F32, m, n, k)
        if all(d[x] == y for x, y in want.items()):
            return bs.TIER_REGISTER | (k << 8)
    raise AssertionError(want)


# both sizes of batch of the register tier's forms, with and without the QR, tall and wide; the shared tier
@pytest.mark.parametrize("m,n,tier", [(54, 45, "reg"), (45, 54, "reg"), (120, 50, "reg"), (64, 64, "precond"),
                                      (64, 64, "carried"), (20, 20, "reg"), (127, 100, "shared"), (30, 90, "shared"),
                                      (24, 9, "shared"), (200, 40, "shared")])
@pytest.mark.parametrize("large", [False, True])
def test_null_entries(m, n, tier, large):
    import paper_1707_05141_gb300 as bs
    bs.build()
    b = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 5 if large else 9
    code = {"reg": lambda: bs.TIER_REGISTER, "shared": lambda: bs.TIER_SHARED,
            "precond": lambda: _variant(bs, m, n, slots=32, qr_precond=1, carried_norms=1),
            "carried": lambda: _variant(bs, m, n, slots=32, qr_precond=0, carried_norms=1)}[tier]()
    k = min(m, n)
    a = torch.randn((b, n, m), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    a *= torch.exp(-torch.arange(n, device="cuda") / 8.0)[None, :, None]

    def run(no_u, no_v):
        s, u, v = (torch.full(z, 7.0, device="cuda") for z in ((b, 1, k), (b, k, m), (b, k, n)))
        info = torch.zeros(b, dtype=torch.int32, device="cuda")
        U, V = bs.Batch.uniform(u, m, k), bs.Batch.uniform(v, n, k)
        U.ptrs[no_u] = 0
        V.ptrs[no_v] = 0
        bs.batched_svd_jacobi(bs.Batch.uniform(a, m, n), bs.Batch.uniform(s, k, 1), U, V, info, tier=code)
        return s, u, v, info

    none = torch.zeros(b, dtype=torch.bool, device="cuda")
    s, u, v, info = run(none, none)
    i = torch.arange(b, device="cuda")
    no_u, no_v = i % 3 == 1, i % 4 >= 2
    s2, u2, v2, info2 = run(no_u, no_v)
    assert torch.equal(s, s2) and torch.equal(info, info2) and bool((info > 0).all())
    assert torch.equal(u2, torch.where(no_u[:, None, None], 7.0, u))
    assert torch.equal(v2, torch.where(no_v[:, None, None], 7.0, v))
