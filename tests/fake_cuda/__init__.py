"""The library's host side on a stand-in CUDA runtime (fake_cuda.cpp): its object
files linked against functions that allocate, launch and copy nothing."""
import ctypes
import importlib.util
import pathlib
import subprocess

import numpy as np

from paper_2012_07620_gb300 import build

HERE = pathlib.Path(__file__).resolve().parent


def load(tmp_path):
    """A copy of the binding on the linked library, its `fake` attribute the
    stand-in's own functions."""
    build.build()
    objs = sorted((build.OUT_DIR / "obj").glob("*.o"))
    if {o.stem for o in objs} != {s.stem for s in build.sources()}:
        build.build(force=True)
        objs = sorted((build.OUT_DIR / "obj").glob("*.o"))
    so = tmp_path / "librerank_fake.so"
    inc = pathlib.Path(build._nvcc()).resolve().parents[1] / "include"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-O1", f"-I{inc}", str(HERE / "fake_cuda.cpp"),
                    *map(str, objs), "-o", str(so), "-Wl,-Bsymbolic", "-lpthread", "-ldl"], check=True)
    spec = importlib.util.spec_from_file_location("rerank_on_fake_cuda", build.PKG / "rerank.py")
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod._LIB_PATH = so
    lib = mod.fake = mod.load_library()
    lib.fake_reset.argtypes = [ctypes.c_size_t]
    lib.fake_count.argtypes, lib.fake_count.restype = [ctypes.c_char_p], ctypes.c_longlong
    for f in (lib.fake_used, lib.fake_peak):
        f.argtypes, f.restype = [ctypes.c_int], ctypes.c_size_t
    return mod


def device(mod, shape, dtype=np.float32):
    """Memory of the stand-in's current device as an array that is passed on, never read."""
    nbytes = int(np.prod(shape)) * np.dtype(dtype).itemsize
    p = ctypes.c_void_p()
    assert mod.fake.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
    return np.ndarray(shape, dtype, buffer=(ctypes.c_char * nbytes).from_address(p.value))
