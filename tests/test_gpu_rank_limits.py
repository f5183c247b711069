"""Ranking by short lists at its limits: queries handed on to the full kernel
while their products are still being added."""
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
        return idx, dist


@pytest.mark.parametrize("ng", [6200, 7000, 24000])  # two CTAs per SM (a score or two past the list, many), one
def test_queries_handed_on_while_they_are_added_up(lib, monkeypatch, ng):
    """Rows without clusters: after three layers a query meets nearly every gallery
    row, so its 16 or 32 warps pass the list's 6,144 places at different moments."""
    nq = 300
    x = torch.randn(nq + ng, 32, generator=torch.Generator().manual_seed(ng)).cuda()
    i0, d0 = _run(lib, monkeypatch, x, nq, 48, 40, 3, ng, short=True)
    i1, d1 = _run(lib, monkeypatch, x, nq, 48, 40, 3, ng, short=False)
    assert ((d0 != 1).sum(1) > 6144).any()
    assert torch.equal(i0, i1) and torch.equal(d0, d1)
