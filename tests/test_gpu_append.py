"""The append pass of the tensor-core similarity stage (sampled floors, segments,
selection) gives the neighbour lists of the FP32 path: at the edges of its
plan (row counts around a tile, around 1,024 where sampling starts, around the
sample sizes' steps), with odd widths, with rows sorted by cluster, and where a
memory budget leaves only room for the list kernels; massive ties (segments run
over) are refused as on the FP32 path."""
import numpy as np
import pytest

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


def _lists(lib, x, k, precision, **kw):
    with lib.Reranker(device=0, precision=precision, **kw) as R:
        idx, score = R.knn(x.cuda(), k)
        torch.cuda.synchronize()
        return idx.cpu().numpy(), score.cpu().numpy(), R.last_info()


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("n,d,k", [(33, 7, 9), (255, 64, 20), (257, 65, 48), (1023, 96, 26), (1024, 128, 26),
                                   (1025, 130, 26), (1281, 64, 48), (4095, 257, 30), (8193, 128, 26),
                                   (16385, 96, 26)])
def test_lists_equal_the_fp32_path(lib, n, d, k, precision):
    x = _clustered(n, d, seed=n)
    fi, fs, _ = _lists(lib, x, k, "fp32")
    bi, bs, info = _lists(lib, x, k, precision)
    assert info["candidates_per_row"] == min(64, n)
    assert (bi == fi).all()
    # Scores: the same bits where both paths pad d alike.  FP8 pads to 128 columns
    # instead of 64, which widens the near-tie rule, so another pair's score may
    # be the FP64 one: both stay within the interface's bound on a score.
    dp = (d + 127) // 128 * 128
    if precision == "bf16" or dp == (d + 63) // 64 * 64:
        assert (bs == fs).all()
    else:
        assert np.abs(bs - fs).max() <= 2 * (dp / 32 + 10) * 2.0 ** -24 * 1.01


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_massive_ties_are_refused_like_the_fp32_path(lib, precision):
    """A few distinct directions, each repeated hundreds of times: every copy ties,
    so floors admit whole classes and segments run over.  No list of 64 candidates
    can bound the rest, which every path reports as EINTERNAL (status 6)."""
    base = _clustered(5, 64, seed=3)
    x = base[torch.randint(5, (2000,), generator=torch.Generator().manual_seed(1))]
    for p in ("fp32", precision):
        with pytest.raises(lib.RerankError) as e:
            _lists(lib, x, 20, p)
        assert e.value.status == 6


def test_sorted_rows(lib):
    """Neighbours stored side by side (rows sorted by cluster) fill few segments."""
    n, d = 6000, 128
    g = torch.Generator().manual_seed(5)
    c = torch.randn(60, d, generator=g)
    x = c.repeat_interleave(100, 0) / d ** 0.5 + 0.4 / d ** 0.5 * torch.randn(n, d, generator=g)
    fi, _, _ = _lists(lib, x, 40, "fp32")
    bi, _, info = _lists(lib, x, 40, "bf16")
    assert (bi == fi).all()


def test_budget_without_room_for_segments(lib):
    x = _clustered(5000, 128, seed=9)
    i0, s0, full = _lists(lib, x, 26, "bf16")
    _, _, small = _lists(lib, x, 26, "bf16", rescore_m=8)
    budget = int(full["workspace_bytes"] * 8 / 9 * 0.8)  # below the append plan, above the list kernels' plan
    i1, s1, info = _lists(lib, x, 26, "bf16", hbm_budget=budget)
    assert info["workspace_bytes"] <= budget and info["candidates_per_row"] == 42
    assert (i1 == i0).all() and (s1 == s0).all()


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_batch_mixes_sampled_and_unsampled_instances(lib, precision):
    with lib.Reranker(device=0, precision=precision) as R, lib.Reranker(device=0, precision=precision) as R1:
        jobs = []
        for n, d in [(60, 64), (900, 64), (1100, 256), (5000, 128), (1024, 512)]:
            x = _clustered(n, d, seed=n + d).cuda()
            jobs.append(dict(xq=x[: n // 7].contiguous(), xg=x[n // 7:].contiguous(), k1=20, k2=6, layers=2))
        outs = R.run_batch(jobs)
        for j, (idx, dist) in zip(jobs, outs):
            i1, d1 = R1.run(j["xq"], j["xg"], 20, 6, 2)
            assert (idx == i1).all() and (dist == d1).all()
