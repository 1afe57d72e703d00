"""The library's objects linked with a fake CUDA runtime (fake_runtime.cpp): no GPU needed."""
import ctypes
import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
NVCC = os.environ.get("NVCC", "nvcc")
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(NVCC) or NVCC))), "include")


def build() -> str:
    from paper_1705_01801_gb300 import build as product
    product.build()
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so, cpp, cu = (os.path.join(out, "libfake.so"), os.path.join(HERE, "fake_runtime.cpp"),
                   os.path.join(HERE, "fake_checks.cu"))
    obj = os.path.join(out, "fake_checks.o")
    objs = sorted(glob.glob(os.path.join(product.OUT, "obj", "*.o")))
    headers = glob.glob(os.path.join(product.CSRC, "*.*h"))
    if product._stale(obj, [cu] + headers):
        subprocess.run([NVCC, *product.ARCH, *product.FLAGS, "-c", cu, "-o", obj], check=True)
    if product._stale(so, [cpp, obj] + objs):
        run = "_ZN3lbw12resident_runEPKNS_8ResidentEPKNS_4GridEPKvRKNS_8ResStateEi"
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CUDA_INCLUDE, "-Wl,-Bsymbolic",
                        "-Wl,--wrap=" + run, cpp, obj, *objs, "-o", so, "-lpthread"], check=True)
    return so


def load():
    """The binding module of the library, on the fake."""
    import importlib.util

    from paper_1705_01801_gb300 import lbw
    spec = importlib.util.spec_from_file_location("paper_1705_01801_gb300._lbw_on_fake", lbw.__file__)
    mod = importlib.util.module_from_spec(spec)
    sys.modules[spec.name] = mod
    spec.loader.exec_module(mod)
    mod._build = type("FakeBuild", (), {"build": staticmethod(build), "SO": ""})
    L = mod.lib()
    L.fake_errors.restype = ctypes.c_char_p
    L.fake_adam_correction.restype = ctypes.c_float
    L.fake_largest_allocation.argtypes = [ctypes.c_size_t]
    return mod
