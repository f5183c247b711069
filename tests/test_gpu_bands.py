"""The append pass over bands of rows that share their segments gives the lists of
one pass over all rows."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_07620_gb300 import rerank
    return rerank


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("n,d", [(257, 64), (1025, 96), (4096, 64), (5889, 200)])
def test_bands_equal_one_pass(lib, monkeypatch, n, d, precision):
    g = torch.Generator().manual_seed(n)
    c = torch.randn(max(1, n // 12), d, generator=g)
    x = (c[torch.randint(len(c), (n,), generator=g)] + 0.5 * torch.randn(n, d, generator=g)).cuda()
    out = []
    for nbytes in (None, "1", "20000000"):  # all rows, 256 rows a band, some bands
        if nbytes:
            monkeypatch.setenv("RERANK_TEST_SEGMENT_BYTES", nbytes)
        with lib.Reranker(device=0, precision=precision) as R:
            out.append((*R.knn(x, 26), R.last_info()["kernel_launches"]))
            torch.cuda.synchronize()
    assert out[1][2] == out[0][2] + 2 * ((n - 1) // 256)  # an append and a selection per band
    for i, s, _ in out[1:]:
        assert torch.equal(i, out[0][0]) and torch.equal(s, out[0][1])
