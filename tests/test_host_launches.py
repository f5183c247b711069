"""Launch shapes at the largest sizes, on a stand-in runtime that refuses a grid or
block beyond the limits of a real launch."""
import pytest

import fake_cuda


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("nq", [4194240, 4194241, 8388480])  # 65,535 tiles of 64 queries, one more, of 128
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_dense_cosines_of_many_queries(lib, nq, precision):
    lib.fake.fake_reset(1 << 42)
    lib.fake.cudaSetDevice(0)
    a = [fake_cuda.device(lib, s) for s in ((nq, 8), (300, 8))]
    oi, od = fake_cuda.device(lib, (nq, 1), "int32"), fake_cuda.device(lib, (nq, 1))
    with lib.Reranker(device=0, precision=precision, rescore_m=4, feature="x") as R:
        R.run(*a, 4, 4, 1, 1, oi, od, stream=0)
    assert lib.fake.fake_count(b"refused") == 0 and lib.fake.fake_count(b"k7_dense_scores") == 1
