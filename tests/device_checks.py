"""Builds tests/device_checks.cu with the library's objects and binds it as the library is bound."""
import ctypes as C
import os
import subprocess


def load(tmp):
    """paper_2207_14256_gb300.fdf on the check library; restore with unload(fdf)."""
    from paper_2207_14256_gb300 import build, fdf

    build.build()
    here = os.path.dirname(os.path.abspath(__file__))
    so = os.path.join(str(tmp), "libchecks.so")
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    objs = [o for o in objs if os.path.basename(o) != "fdf_api.o"]
    cmd = [build._nvcc(), *build.ARCH, *build.FLAGS, "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
           "-shared", "-o", so, os.path.join(here, "device_checks.cu"), *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    fdf._lib, fdf.LIB_PATH = None, so
    L = fdf.lib()
    L.fdf_check_grid.argtypes = [C.c_void_p, C.c_int32, C.c_void_p, C.c_size_t]
    L.fdf_check_kick_fp64.argtypes = [C.c_int32, C.POINTER(C.c_int32)]
    L.fdf_check_kick_fp64.restype = None
    L.fdf_check_bits.argtypes = [C.c_int64] + [C.c_void_p] * 4
    return fdf


def unload(fdf):
    fdf._lib, fdf.LIB_PATH = None, os.path.join(fdf.HERE, "libfdf.so")
