"""Selections whose buckets or segments run over, against FP64: one tight cluster
(hundreds of scores in one bucket of the selection kernels), and rows along a
curve (a row's neighbours side by side, more of them than a segment holds)."""
import json
import math

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

INVALID = 0x7FFFFFFF


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2012_07620_gb300 import rerank
    return rerank


def _exact(x, k):
    """Top-k lists in FP64, self first (its score counts as 1)."""
    u = x.double()
    u = u / u.norm(dim=1, keepdim=True)
    idx, val = [], []
    for a in range(0, len(u), 4096):
        s = u[a:a + 4096] @ u.T
        s[torch.arange(len(s)), torch.arange(a, a + len(s))] = 1.0
        v, i = s.topk(k, dim=1)
        idx.append(i)
        val.append(v)
    return torch.cat(idx), torch.cat(val)


def _check(lib, x, k, precision, **kw):
    """The lists equal FP64's; the approximate lists and the counters of the call."""
    n, d = x.shape
    with lib.Reranker(device=0, precision=precision, **kw) as R:
        idx, score = R.knn(x, k)
        torch.cuda.synchronize()
        info = R.last_info()
        part = [torch.from_numpy(R.debug(w)).reshape(n, -1) for w in ("part_s", "part_i")]
    ri, rs = _exact(x, k)
    assert torch.equal(idx.long(), ri)
    dp = -(-d // 128) * 128
    assert (score.double() - rs).abs().max() <= (dp / 32 + 10) * 2.0 ** -24 * 1.01
    return part, info


def _tight_cluster(n, d):
    """Groups of ten (cosine 0.9995 inside) around one direction (0.987 between groups)."""
    g = torch.Generator().manual_seed(6)
    groups = torch.randn(n // 10 + 1, d, generator=g).repeat_interleave(10, 0)[:n]
    x = torch.randn(1, d, generator=g) + math.sqrt(0.0125) * groups + math.sqrt(0.0005) * torch.randn(n, d, generator=g)
    return x[torch.randperm(n, generator=g)].cuda()


@pytest.mark.parametrize("n", [900, 3000, 6010])  # every column kept, sampled
def test_crowded_bucket_of_the_tensor_core_selection(lib, n):
    x = _tight_cluster(n, 256)
    (ps, pi), info = _check(lib, x, 8, "bf16")
    assert info["fallback_rows"] == 0  # certified from the selection's lists
    # Those are the 64 best by the approximate scores (of the BF16 rows, to FP32 accumulation).
    u = (x * (1 / x.double().norm(dim=1, keepdim=True)).float()).bfloat16().double()
    s = u @ u.T
    s.fill_diagonal_(1.0)
    listed = s.gather(1, pi.cuda().long())
    assert (listed - ps.cuda().double()).abs().max() <= 2e-5
    assert (listed.min(1).values >= s.topk(64, dim=1).values[:, -1] - 2e-5).all()
    assert (ps[:, 1:] <= ps[:, :-1]).all()
    assert all(len(set(r)) == 64 for r in pi[::97].tolist())
    # more than 128 scores down to the end of the 64th one's bucket, [126 / 128, 127 / 128)
    v = s.topk(64, dim=1).values[:, -1]
    assert v.max() < 127 / 128 and v.min() > 126 / 128 and (s > 126 / 128).sum(1).min() > 128


@pytest.mark.parametrize("n", [900, 3000, 6010])
def test_crowded_bucket_of_the_fp32_selection(lib, n):
    _check(lib, _tight_cluster(n, 256), 30, "fp32")


@pytest.mark.parametrize("chunks", [0, 16])  # of the work split's own: segments of 256 places; 128
@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_segments_that_run_over(lib, tmp_path, precision, chunks):
    """cos(t, t + e) = exp(-(e / 150)^2 / 2): a row's some 450 admitted columns lie
    side by side, over 100 of them in the same segment, which takes no more within
    32 places of its end."""
    n, d = 32700, 1030
    g = torch.Generator().manual_seed(7)
    t = torch.arange(n, dtype=torch.float64)[:, None]
    x = torch.cos(t * torch.randn(1, d, generator=g, dtype=torch.float64) / 150
                  + 2 * math.pi * torch.rand(1, d, generator=g, dtype=torch.float64))
    x = (x + 0.01 * torch.randn(n, d, generator=g, dtype=torch.float64)).float().cuda()
    table = tmp_path / "tune.json"
    table.write_text(json.dumps({"version": 1, "entries": [
        {"precision": lib.PRECISION[precision], "d": d, "n_bucket": int(2 * math.log2(n)), "sim_chunks": chunks,
         "prop_warps": 8, "refine_order": 1, "ms": 1.0}]}))
    (_, pi), info = _check(lib, x, 26, precision, autotune_path=str(table))
    over = (pi[:, 0] == INVALID).sum()
    assert (over > 0) == (chunks == 16) and info["fallback_rows"] >= over
