"""The bench names the kernel that its tier launches."""
import bench
import paper_1707_05141_gb300 as bs


def test_jacobi_kernel_of_a_tier():
    seen = set()
    for k in range(1, bs.jacobi_variants(bs.F32, 64, 64, bs.TIER_REGISTER) + 1):
        d = bs.jacobi_variant_desc(bs.F32, 64, 64, k)
        separate = d["slots"] == 32 and d["rows_a"] == 32 and d["scaled"]
        name = bench.jacobi_kernel(bs, bs.F32, 64, 64, bs.TIER_REGISTER | k << 8)
        assert name == ("jacobi_wv_kernel" if separate else "jacobi_reg_kernel"), d
        seen.add(name)
    assert len(seen) == 2
    assert bench.jacobi_kernel(bs, bs.F64, 32, 32, bs.TIER_REGISTER) == "jacobi_reg_kernel"
    assert bench.jacobi_kernel(bs, bs.F32, 64, 64, bs.TIER_SHARED) == "jacobi_rx_kernel"
    assert bench.jacobi_kernel(bs, bs.F32, 64, 16, bs.TIER_SHARED) == "jacobi_rx8_kernel"
    assert bench.jacobi_kernel(bs, bs.F32, 200, 64, bs.TIER_SHARED) == "jacobi_smem_kernel"
    assert bench.jacobi_kernel(bs, bs.F64, 64, 64, bs.TIER_SHARED) == "jacobi_smem_kernel"
