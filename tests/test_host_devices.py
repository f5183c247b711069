"""Every device of a process gets working launches: contexts on two devices, one
after the other, on a stand-in runtime that keeps a kernel's shared-memory limit
per device as the real one does."""
import pytest

import fake_cuda


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


def _run_on(lib, device, precision, n=1500, ng=1400):
    lib.fake.cudaSetDevice(device)
    nq, d = n - ng, 96
    a = [fake_cuda.device(lib, s) for s in ((nq, d), (ng, d))]
    oi, od = fake_cuda.device(lib, (nq, ng), "int32"), fake_cuda.device(lib, (nq, ng))
    with lib.Reranker(device=device, precision=precision) as R:
        R.run(*a, 26, 7, 2, 0, oi, od, stream=0)


@pytest.mark.parametrize("precision", ["fp32"])
def test_second_device_of_a_process(lib, precision):
    lib.fake.fake_reset(1 << 36)
    for device in (0, 1, 0):
        _run_on(lib, device, precision)
    assert lib.fake.fake_count(b"refused") == 0
