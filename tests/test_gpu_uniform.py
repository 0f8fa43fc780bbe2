"""The pointer and size arrays of a uniform batch, written by one kernel, against the arithmetic they stand for."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("batch,cols,ld,m,n", [(0, 3, 4, None, None), (1, 1, 1, None, None), (127, 20, 33, 30, 7),
                                               (128, 5, 6, 1, 1), (129, 2, 3, None, 2), (5, 0, 4, None, None)])
def test_arrays(dtype, batch, cols, ld, m, n):
    import paper_1707_05141_gb300 as bs
    bs.build()
    t = torch.zeros((batch, cols, ld), device="cuda", dtype=dtype)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        b = bs.Batch.uniform(t, m, n)
    stream.synchronize()
    m, n = ld if m is None else m, cols if n is None else n
    assert b.ptrs.tolist() == [t.data_ptr() + i * cols * ld * t.element_size() for i in range(batch)]
    assert b.m.tolist() == [m] * batch and b.n.tolist() == [n] * batch and b.ld.tolist() == [ld] * batch
    assert (b.batch, b.max_m, b.max_n) == (batch, m, n)
    assert b.ptrs.dtype == torch.int64 and {b.m.dtype, b.n.dtype, b.ld.dtype} == {torch.int32}


def test_refused():
    import paper_1707_05141_gb300 as bs
    bs.build()
    with pytest.raises(TypeError):
        bs.Batch.uniform(torch.zeros((2, 3, 4), device="cuda", dtype=torch.float16))
    with pytest.raises(ValueError):
        bs.Batch.uniform(torch.zeros((2, 3, 4)))
    with pytest.raises(ValueError):
        bs.Batch.uniform(torch.zeros((2, 3, 4), device="cuda").transpose(1, 2))
