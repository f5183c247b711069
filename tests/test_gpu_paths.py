"""Kernels chosen by size or memory give the results of the ones they stand in
for: the FP32 similarity from the symmetric matrix and from streamed lists, the
rows of unaligned inputs normalised in registers, queries ranked by short lists
and by the full kernel, and served requests that read the resident graph's rows
in place for every aggregator, feature and depth."""
import numpy as np
import pytest

import parity
from oracle import rerank_oracle as o
from paper_2012_07620_gb300 import synthetic

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_07620_gb300 import rerank
    return rerank


def _clustered(n, d, seed, sigma=0.5):
    g = torch.Generator().manual_seed(seed)
    c = torch.randn(max(1, n // 12), d, generator=g)
    x = c[torch.randint(len(c), (n,), generator=g)]
    return x / x.norm(dim=1, keepdim=True) + sigma / d ** 0.5 * torch.randn(n, d, generator=g)


def _knn(lib, x, k, **kw):
    with lib.Reranker(device=0, **kw) as R:
        idx, score = R.knn(x.cuda(), k)
        torch.cuda.synchronize()
        return idx.cpu().numpy(), score.cpu().numpy(), R.last_info()


@pytest.mark.parametrize("n,d,k", [(5889, 64, 26), (6016, 130, 48), (6017, 65, 1)])
def test_fp32_matrix_and_streamed_lists_agree(lib, n, d, k):
    """Row counts around a multiple of the matrix's 128-row tiles.  Both paths
    compute a score by the same chain of FMAs: equal lists, equal bits."""
    x = _clustered(n, d, seed=n)
    i0, s0, full = _knn(lib, x, k, precision="fp32")
    budget = full["workspace_bytes"] - 2 * n * n  # half the matrix
    i1, s1, info = _knn(lib, x, k, precision="fp32", hbm_budget=budget)
    assert info["workspace_bytes"] <= budget
    assert (i1 == i0).all() and (s1 == s0).all()


@pytest.mark.parametrize("n,d,k", [(2, 8, 1), (127, 64, 9), (128, 36, 20), (129, 64, 48), (700, 100, 26)])
def test_fp32_matrix_equals_tensor_core_lists(lib, n, d, k):
    x = _clustered(n, d, seed=n)
    i0, _, _ = _knn(lib, x, k, precision="fp32")
    i1, _, _ = _knn(lib, x, k, precision="bf16")
    assert (i1 == i0).all()


@pytest.mark.parametrize("d", [1, 31, 64, 127, 512, 513, 1024, 2047, 2048, 2052])
def test_bf16_rows_equal_their_fp32_values(lib, d):
    """The register kernel (BF16 rows, odd widths) up to 2,048 columns, the
    general one beyond: the same values enter, so the lists are equal and the
    scores are, within the interface's bound on each."""
    x = _clustered(300, d, seed=d).bfloat16()
    wide = torch.zeros(300, (d + 3) // 4 * 4)  # 16-byte rows: the vector kernel
    wide[:, :d] = x.float()
    eps = ((d + 63) // 64 * 64 / 32 + 10) * 2.0 ** -24 * 1.01
    if d == 1:  # every score is +-1: more ties than the FP32 path's candidates, refused for either input
        for v in (x[:40], wide[:40]):
            with pytest.raises(lib.RerankError) as err:
                _knn(lib, v, 4, precision="fp32")
            assert err.value.status == 6
        return
    i0, s0, _ = _knn(lib, x, 20, precision="fp32")
    i1, s1, _ = _knn(lib, wide, 20, precision="fp32")
    assert (i0 == i1).all() and np.abs(s0 - s1).max() <= 2 * eps


@pytest.mark.parametrize("nq,ng,k1,k2,layers,topk", [
    (3, 61, 8, 3, 2, 0), (40, 500, 20, 6, 2, 0), (40, 500, 20, 6, 2, 7), (33, 2000, 26, 7, 2, 2000),
    (64, 9000, 48, 40, 3, 0),      # most queries have more non-zeros than a short list holds
    (20, 19700, 26, 7, 2, 0), (20, 20100, 26, 7, 2, 100),  # two CTAs per SM, one
    (20, 46000, 26, 7, 2, 100)])   # past the short lists' shared memory
def test_short_lists_rank_like_the_full_kernel(lib, monkeypatch, nq, ng, k1, k2, layers, topk):
    x = _clustered(nq + ng, 64, seed=ng).cuda()
    out = []
    for caps in (None, "8191,256"):  # a lowered cap of the full kernel's sort turns the short lists off
        if caps:
            monkeypatch.setenv("RERANK_TEST_RANK_CAPS", caps)
        with lib.Reranker(device=0, precision="bf16") as R:
            idx, dist = R.run(x[:nq].contiguous(), x[nq:].contiguous(), k1, k2, layers, topk or ng)
            torch.cuda.synchronize()
            out.append((idx.cpu().numpy(), dist.cpu().numpy()))
    assert (out[0][0] == out[1][0]).all() and (out[0][1] == out[1][1]).all()


@pytest.mark.parametrize("layers,aggregator,feature,k1,k2", [
    (0, "sum", "astar", 26, 7), (1, "max", "astar", 26, 7), (3, "mean", "astar", 20, 5), (2, "sum", "a", 26, 7),
    (2, "sum", "astar", 40, 34)])  # more messages than lanes
def test_served_rows_in_place(lib, layers, aggregator, feature, k1, k2):
    """As a fresh run on the union: distances to 1e-6 (the bound of the serving
    tests), places swapped only where distances tie to that."""
    spec = synthetic.WorkloadSpec("serve_paths", 0, 1500, 128, 90, 0.35, 0, None, seed=5)
    w = synthetic.make_workload(spec)
    xg = torch.from_numpy(w.xg).cuda()
    kw = dict(precision="bf16", aggregator=aggregator, feature=feature)
    with lib.Reranker(**kw) as R, lib.Reranker(**kw) as F:
        R.load_gallery(xg, max_query=64, k1=k1, k2=k2, layers=layers, slots=2)
        for r, nq in enumerate((1, 33, 64)):
            q = torch.from_numpy(synthetic.request_queries(w, 50 + r, nq)).cuda()
            t, si, sd = R.submit(q, 0)
            assert R.wait(t, 120000) is not None
            fi, fd = F.run(q, xg, k1, k2, layers)
            torch.cuda.synchronize()
            si, sd, fi, fd = (v.cpu().numpy() for v in (si, sd, fi, fd))
            assert np.abs(sd.astype(np.float64) - fd).max() <= 1e-6
            differ = si != fi
            assert np.all(np.abs(sd[differ].astype(np.float64) - fd[differ]) <= 1e-6)


@pytest.mark.parametrize("ng", [8191, 8192, 8200])
def test_column_lists_by_cta_equal_the_oracle(lib, ng):
    """The gallery's column lists from 8,192 rows up are counted per CTA."""
    spec = synthetic.WorkloadSpec("columns", 12, ng, 64, 400, 0.35, 0, None, seed=7)
    w = synthetic.make_workload(spec)
    ref = o.rerank(w.xq, w.xg, k1=20, k2=5, layers=2, mode="sparse")
    with lib.Reranker(device=0, precision="bf16") as R:
        idx, dist = R.run(torch.from_numpy(w.xq).cuda(), torch.from_numpy(w.xg).cuda(), 20, 5, 2)
        torch.cuda.synchronize()
    parity.assert_ranked_equal(idx.cpu().numpy(), dist.cpu().numpy(), ref.s, ref.idx)


@pytest.mark.parametrize("ng", [8191, 8192])
def test_gallery_column_lists_at_load(lib, ng):
    """The resident graph's column lists, built at load, from 8,192 rows up per CTA."""
    spec = synthetic.WorkloadSpec("load_columns", 0, ng, 64, 400, 0.35, 0, None, seed=9)
    w = synthetic.make_workload(spec)
    xg = torch.from_numpy(w.xg).cuda()
    q = torch.from_numpy(synthetic.request_queries(w, 3, 5)).cuda()
    with lib.Reranker(precision="bf16") as R, lib.Reranker(precision="bf16") as F:
        R.load_gallery(xg, max_query=16, k1=20, k2=5, layers=2, slots=2)
        t, si, sd = R.submit(q, 0)
        assert R.wait(t, 120000) is not None
        assert R.serve_info()["reuse_layers"] == 1
        fi, fd = F.run(q, xg, 20, 5, 2)
        torch.cuda.synchronize()
        si, sd, fi, fd = (v.cpu().numpy() for v in (si, sd, fi, fd))
    assert np.abs(sd.astype(np.float64) - fd).max() <= 1e-6
    differ = si != fi
    assert np.all(np.abs(sd[differ].astype(np.float64) - fd[differ]) <= 1e-6)
