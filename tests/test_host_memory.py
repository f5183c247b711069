"""Plans at the limits of device memory, on a stand-in runtime with a set capacity:
which plan a call ends up with, and what it allocates and frees."""
import pytest

import fake_cuda

MB = 1 << 20


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


class Case:
    """One instance in the stand-in's memory, and what its two plans take."""

    def __init__(self, lib, precision, n=20000, d=128, nq=500, jobs=1):
        lib.fake.fake_reset(1 << 40)
        lib.fake.cudaSetDevice(0)
        self.lib, self.precision = lib, precision
        x = fake_cuda.device(lib, (n, d))
        self.x, self.nq = x, nq
        self.jobs = [dict(xq=x[:nq], xg=x[nq:], k1=26, k2=7, layers=2, topk_out=100,
                          out_idx=fake_cuda.device(lib, (nq, 100), "int32"),
                          out_dist=fake_cuda.device(lib, (nq, 100))) for _ in range(jobs)]
        self.base = lib.fake.fake_used(0)
        with self.context() as R:
            self.call(R)
            self.wide = R.last_info()["workspace_bytes"] * 8 // 9  # allocations have an eighth to spare
        with self.context(hbm_budget=self.wide - 1) as R:
            self.call(R)
            self.narrow = R.last_info()["workspace_bytes"]
        assert self.narrow + 16 * MB < self.wide

    def context(self, **kw):
        return self.lib.Reranker(device=0, precision=self.precision, **kw)

    def call(self, R):
        if len(self.jobs) > 1:
            R.run_batch(self.jobs, stream=0)
        else:
            j = self.jobs[0]
            R.run(j["xq"], j["xg"], 26, 7, 2, 100, j["out_idx"], j["out_dist"], stream=0)

    def room(self, nbytes):
        self.lib.fake.fake_reset(self.base + nbytes + MB)  # the status block and the like

    def allocations(self):
        return [self.lib.fake.fake_count(w) for w in (b"cudaMalloc", b"cudaFree")]


@pytest.mark.parametrize("precision,jobs", [("fp32", 1), ("bf16", 1), ("fp8", 1), ("fp32", 3), ("bf16", 3)])
def test_a_plan_without_room_is_not_tried_again(lib, precision, jobs):
    c = Case(lib, precision, jobs=jobs)
    c.room(c.narrow)
    with c.context() as R:
        c.call(R)
        first = c.allocations()
        for _ in range(4):
            c.call(R)
        assert c.allocations() == first
        if jobs > 1:  # captured by the second call and replayed, not dropped
            assert lib.fake.fake_count(b"graph captured") == 1
            assert lib.fake.fake_count(b"graph launched") == 4


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_the_exact_size_is_tried_before_a_plan_is_given_up(lib, precision):
    c = Case(lib, precision)
    c.room(c.wide)
    with c.context() as R:
        c.call(R)
        assert c.narrow < R.last_info()["workspace_bytes"] <= c.wide + MB


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_segments_of_a_large_instance_are_bounded(lib, precision):
    """At most 4 GB beside the plan with lists (64 KB a row otherwise: 65 GB here)."""
    lib.fake.fake_reset(1 << 40)
    n = 1000000
    x, oi, os = (fake_cuda.device(lib, (n, w), t) for w, t in ((64, "f4"), (26, "i4"), (26, "f4")))
    with lib.Reranker(device=0, precision=precision) as R:
        R.knn(x, 26, oi, os, stream=0)
        need = R.last_info()["workspace_bytes"] * 8 // 9
    recheck = n * 32 * 64 * 8  # its lists, the largest buffer of either plan
    assert need < recheck + (4 << 30) + (3 << 30)  # rows, copies and the final lists


@pytest.mark.parametrize("precision,n,jobs", [("fp32", 20000, 40), ("bf16", 8000, 160)])
def test_a_batch_takes_no_more_than_its_share_for_speed(lib, precision, n, jobs):
    """16 GB of matrices and segments for the call, not for each instance (64 and 21 GB here)."""
    c = Case(lib, precision, n=n, jobs=jobs)
    assert c.wide <= c.narrow + (16 << 30) + jobs * MB


@pytest.mark.parametrize("n,d,k,m", [(724988, 7, 27, 0), (458472, 7, 38, 16)])
def test_large_lists_in_little_memory(lib, n, d, k, m):
    """8 GB hold these lists where a row has no more of them than the work split wants."""
    lib.fake.fake_reset(1 << 40)
    x, oi, os = (fake_cuda.device(lib, (n, w), t) for w, t in ((d, "f4"), (k, "i4"), (k, "f4")))
    with lib.Reranker(device=0, precision="bf16", rescore_m=m, hbm_budget=8 << 30) as R:
        R.knn(x, k, oi, os, stream=0)
