"""Kernels chosen by size, at the limits of the choice: ranking by short lists
(queries handed on to the full kernel while their products are still being added;
the last gallery that fits beside the lists, twice per SM and once), and the FP32
similarity with and without its matrix."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_07620_gb300 import rerank
    return rerank


def _run(lib, monkeypatch, x, nq, k1, k2, layers, topk, short):
    # a lowered cap of the full kernel's sort turns the short lists off
    monkeypatch.delenv("RERANK_TEST_RANK_CAPS", raising=False)
    if not short:
        monkeypatch.setenv("RERANK_TEST_RANK_CAPS", "8191,256")
    with lib.Reranker(device=0, precision="bf16") as R:
        idx, dist = R.run(x[:nq].contiguous(), x[nq:].contiguous(), k1, k2, layers, topk)
        torch.cuda.synchronize()
        return idx, dist, R.last_info()["kernel_launches"]


@pytest.mark.parametrize("ng", [6200, 7000, 24000])  # two CTAs per SM (a score or two past the list, many), one
def test_queries_handed_on_while_they_are_added_up(lib, monkeypatch, ng):
    """Rows without clusters: after three layers a query meets nearly every gallery
    row, so its 16 or 32 warps pass the list's 6,144 places at different moments."""
    nq = 300
    x = torch.randn(nq + ng, 32, generator=torch.Generator().manual_seed(ng)).cuda()
    i0, d0, _ = _run(lib, monkeypatch, x, nq, 48, 40, 3, ng, short=True)
    i1, d1, _ = _run(lib, monkeypatch, x, nq, 48, 40, 3, ng, short=False)
    assert ((d0 != 1).sum(1) > 6144).any()
    assert torch.equal(i0, i1) and torch.equal(d0, d1)


@pytest.mark.parametrize("ng,short", [(20072, 1), (20073, 1), (48372, 1), (48373, 0)])
def test_last_galleries_of_the_short_lists(lib, monkeypatch, ng, short):
    """227 KB hold the lists and the scores of 48,372 rows, 228 those of two CTAs of 20,072."""
    nq, d = 20, 64
    g = torch.Generator().manual_seed(ng)
    c = torch.randn(ng // 12, d, generator=g)
    x = (c[torch.randint(len(c), (nq + ng,), generator=g)] + 0.5 * torch.randn(nq + ng, d, generator=g)).cuda()
    i0, d0, n0 = _run(lib, monkeypatch, x, nq, 26, 7, 2, ng, short=True)
    i1, d1, n1 = _run(lib, monkeypatch, x, nq, 26, 7, 2, ng, short=False)
    assert n0 - n1 == short
    assert torch.equal(i0, i1) and torch.equal(d0, d1)


@pytest.mark.parametrize("n,d,k", [(5889, 64, 26), (6016, 130, 48), (6017, 65, 1)])
def test_fp32_without_its_matrix(lib, n, d, k):
    x = torch.randn(n, d, generator=torch.Generator().manual_seed(n)).cuda()
    matrix = (-(-n // 128) * 128) ** 2 * 4
    with lib.Reranker(device=0, precision="fp32") as R:
        i0, s0 = R.knn(x, k)
        torch.cuda.synchronize()
        need = R.last_info()["workspace_bytes"] * 8 // 9
    with lib.Reranker(device=0, precision="fp32", hbm_budget=need - 1) as R:
        i1, s1 = R.knn(x, k)
        torch.cuda.synchronize()
        assert R.last_info()["workspace_bytes"] < matrix < need
    assert torch.equal(i0, i1) and torch.equal(s0, s1)
