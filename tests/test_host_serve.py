"""How a gallery is loaded at the limits of memory, on a stand-in runtime with a set
capacity: the plan with full lists and segments gives way to the one without."""
import ctypes

import pytest

import fake_cuda

MB = 1 << 20


class Gallery:
    """A gallery in the stand-in's memory and the least budget that loads it."""

    def __init__(self, lib):
        lib.fake.fake_reset(1 << 40)
        lib.fake.cudaSetDevice(0)
        self.lib = lib
        self.x = fake_cuda.device(lib, (20000, 256))
        self.base = lib.fake.fake_used(0)
        lo, hi = MB, 1 << 40
        while hi - lo > MB // 4:
            mid = (lo + hi) // 2
            if self.load(hbm_budget=mid):
                hi = mid
            else:
                lo = mid
        self.least = hi
        self.slot = self.load(hbm_budget=hi)["slot_bytes"]

    def load(self, slots=8, **kw):
        """What serve_info says, None without room."""
        with self.lib.Reranker(device=0, precision="bf16", **kw) as R:
            try:
                R.load_gallery(self.x, 128, 26, 7, 2, slots=slots)
            except self.lib.RerankError as e:
                assert e.status in (2, 3)
                return None
            return R.serve_info()


@pytest.fixture(scope="module")
def gallery(tmp_path_factory):
    return Gallery(fake_cuda.load(tmp_path_factory.mktemp("fake")))


def test_roomy_memory_takes_the_plan_with_full_lists(gallery):
    gallery.lib.fake.fake_reset(1 << 40)
    info = gallery.load()
    assert info["slots"] == 8 and info["slot_bytes"] > gallery.slot and info["reuse_layers"] == 1


def test_memory_for_the_smaller_plan_is_enough(gallery):
    gallery.lib.fake.fake_reset(gallery.base + gallery.least + MB)
    info = gallery.load()
    assert info and info["slots"] == 1 and info["slot_bytes"] == gallery.slot
    assert gallery.lib.fake.fake_used(0) == gallery.base  # all given back


@pytest.mark.parametrize("slots", [2, 3, 5, 7, 8])
def test_no_slot_is_given_up_for_the_larger_plan(gallery, slots):
    nbytes = gallery.least + (slots - 1) * gallery.slot
    gallery.lib.fake.fake_reset(1 << 40)
    assert gallery.load(hbm_budget=nbytes)["slots"] == slots
    gallery.lib.fake.fake_reset(gallery.base + nbytes + MB)
    assert gallery.load()["slots"] == slots


def test_the_resident_graph_is_not_given_up_for_the_larger_plan(gallery):
    gallery.lib.fake.fake_reset(1 << 40)
    wide = gallery.load(slots=1)
    nbytes = gallery.least + 8 * MB  # the smaller plan, one slot and its graph (some 3 MB here)
    while (info := gallery.load(slots=1, hbm_budget=nbytes))["slot_bytes"] < wide["slot_bytes"]:
        assert info["reuse_layers"] == 1
        nbytes += MB
    assert info["reuse_layers"] == 1  # the first budget that the larger plan is taken with


@pytest.mark.parametrize("precision,ng,d,m,k1,k2,layers,max_query,slots", [
    ("fp8", 404302, 713, 0, 36, 2, 2, 64, 1), ("bf16", 503430, 187, 16, 2, 2, 4, 500, 2),
    ("fp8", 228312, 335, 4, 32, 5, 3, 1024, 2), ("fp8", 225405, 1, 100, 7, 3, 0, 64, 3)])
def test_large_galleries_in_32_gigabytes(gallery, precision, ng, d, m, k1, k2, layers, max_query, slots):
    lib = gallery.lib
    lib.fake.fake_reset(1 << 40)
    x = fake_cuda.device(lib, (ng, d))
    lib.fake.fake_reset(lib.fake.fake_used(0) + (32 << 30) - ng * d * 4)
    with lib.Reranker(device=0, precision=precision, rescore_m=m) as R:
        R.load_gallery(x, max_query, k1, k2, layers, slots=8)
        info = R.serve_info()
        assert info["slots"] >= slots and info["reuse_layers"] == 1
    lib.fake.cudaFree(ctypes.c_void_p(x.ctypes.data))
