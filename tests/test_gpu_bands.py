"""Plans that share or lack the memory the fastest ones take give the same results:
the append pass over bands of rows that share their segments, and batches whose
later instances do without segments or matrix."""
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


@pytest.mark.parametrize("precision,nbytes", [("fp32", 50 << 20), ("bf16", 40 << 20), ("fp8", 40 << 20)])
def test_batch_with_and_without_segments_or_matrix(lib, monkeypatch, precision, nbytes):
    g = torch.Generator().manual_seed(4)
    jobs = []
    for n, d in [(2000, 64), (900, 130), (2600, 256), (3000, 64), (60, 64)]:
        x = (torch.randn(n // 12, d, generator=g)[torch.randint(n // 12, (n,), generator=g)]
             + 0.5 * torch.randn(n, d, generator=g)).cuda()
        jobs.append(dict(xq=x[: n // 7].contiguous(), xg=x[n // 7:].contiguous(), k1=20, k2=6, layers=2))
    out, need = [], []
    for limit in (None, nbytes, 1):  # all instances, some, none
        if limit:
            monkeypatch.setenv("RERANK_TEST_SIDE_BYTES", str(limit))
        with lib.Reranker(device=0, precision=precision) as R:
            for _ in range(2):  # the second call is captured
                res = R.run_batch(jobs)
                torch.cuda.synchronize()
            out.append(res)
            need.append(R.last_info()["workspace_bytes"])
    assert len(set(need)) == 3
    for res in out[1:]:
        for (i, d), (i0, d0) in zip(res, out[0]):
            assert torch.equal(i, i0) and torch.equal(d, d0)


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_large_lists_with_less_and_less_memory(lib, precision):
    """304 column tiles in one chunk: the append pass, lists on pairs (two chunks of
    columns), and lists on single CTAs (one) as the budget shrinks."""
    n, d, k = 77800, 64, 10
    g = torch.Generator(device="cuda").manual_seed(8)
    c = torch.randn(n // 12, d, generator=g, device="cuda")
    x = c[torch.randint(len(c), (n,), generator=g, device="cuda")]
    x += 0.5 * torch.randn(n, d, generator=g, device="cuda")
    budget, out, need = 0, [], []
    for _ in range(4):  # (the first allocation within a new plan has an eighth to spare)
        with lib.Reranker(device=0, precision=precision, hbm_budget=budget) as R:
            out.append(R.knn(x, k))
            torch.cuda.synchronize()
            need.append(R.last_info()["workspace_bytes"])
        budget = (need[-1] * 8 // 9 if len(need) == 1 else need[-1]) - 1
    assert need == sorted(need, reverse=True) and len(set(need)) == 4
    for i, s in out[1:]:
        assert torch.equal(i, out[0][0]) and torch.equal(s, out[0][1])
