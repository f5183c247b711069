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


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp8"])
def test_second_device_of_a_process(lib, precision):
    lib.fake.fake_reset(1 << 36)
    for device in (0, 1, 0):
        _run_on(lib, device, precision)
    assert lib.fake.fake_count(b"refused") == 0


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
def test_batch_and_serving_on_both_devices(lib, precision):
    lib.fake.fake_reset(1 << 38)
    for device in (0, 1):
        lib.fake.cudaSetDevice(device)
        x = fake_cuda.device(lib, (5000, 96))
        oi, od = fake_cuda.device(lib, (64, 100), "int32"), fake_cuda.device(lib, (64, 100))
        with lib.Reranker(device=device, precision=precision) as R:
            job = dict(xq=x[:64], xg=x[64:], k1=26, k2=7, layers=2, topk_out=100, out_idx=oi, out_dist=od)
            R.run_batch([job, job], stream=0)
            R.load_gallery(x, 64, 26, 7, 2, slots=2)
            R.wait(R.submit(x[:64], 100, oi, od, stream=0)[0])
    assert lib.fake.fake_count(b"refused") == 0


def test_no_launch_lowers_a_kernels_shared_memory_limit(lib):
    """The limit is the kernel's, not the launch's: lowering it for a small call would
    fail the larger launch that another thread is about to make."""
    lib.fake.fake_reset(1 << 38)
    for precision in ("fp32", "bf16"):
        for n, ng in ((24000, 23000), (16000, 15000), (1500, 1400)):
            _run_on(lib, 0, precision, n, ng)
    assert lib.fake.fake_count(b"lowered") == 0
