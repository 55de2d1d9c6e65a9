"""The library's host side without a GPU: its objects linked with
cpu_exec/fake_cudart.cpp instead of the CUDA runtime (one shared library of
its own, never the one that the package loads)."""
import ctypes
import glob
import os
import subprocess

from paper_1011_4046_gb300 import build, sp

HERE = os.path.dirname(os.path.abspath(__file__))


def load():
    build.build(force=not all(os.path.exists(os.path.join(build.BUILD, f + ".o")) for f in build.SOURCES))
    out_dir = os.path.join(HERE, "cpu_exec", "_build")
    os.makedirs(out_dir, exist_ok=True)
    lib = os.path.join(out_dir, "libsp_fake.so")
    src = os.path.join(HERE, "cpu_exec", "fake_cudart.cpp")
    objs = sorted(o for o in glob.glob(os.path.join(build.BUILD, "*.o")) if os.path.basename(o)[:-2] in build.SOURCES)
    if not os.path.exists(lib) or any(os.path.getmtime(f) > os.path.getmtime(lib) for f in [src, *objs]):
        tmp = lib + f".tmp{os.getpid()}"
        include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
        subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", f"-I{include}", src, *objs,
                        "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", tmp], check=True)
        os.replace(tmp, lib)
    L = ctypes.CDLL(lib)
    vp, size = ctypes.c_void_p, ctypes.c_size_t
    L.fake_reset.argtypes = [size, ctypes.c_int, ctypes.c_uint]
    L.fake_set_capacity.argtypes = [size]
    L.fake_used.restype = L.fake_peak.restype = size
    L.fake_copies.argtypes = [size, ctypes.POINTER(vp), ctypes.c_int]
    L.sp_grid_create.argtypes = [ctypes.POINTER(sp.sp_params), ctypes.c_int32, ctypes.POINTER(vp), vp, ctypes.POINTER(vp)]
    L.sp_region_plan.argtypes = [vp, ctypes.c_int32, ctypes.c_int32, ctypes.c_int32, ctypes.c_char_p]
    L.sp_evolve.argtypes = [vp, ctypes.c_int64, ctypes.c_uint32]
    L.sp_read_surface.argtypes = [vp, ctypes.c_int32, ctypes.c_int32, vp, size, ctypes.c_int32]
    L.sp_set_option.argtypes = [vp, ctypes.c_int32, ctypes.c_int64]
    L.sp_destroy.argtypes = [vp]
    fp = ctypes.POINTER(ctypes.c_float)
    L.sp_model_create.argtypes = [ctypes.c_uint64, vp, ctypes.POINTER(vp)]
    L.sp_model_destroy.argtypes = [vp]
    L.sp_model_train.argtypes = [vp, vp, vp, ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, ctypes.c_float,
                                 ctypes.c_uint64, ctypes.POINTER(ctypes.c_int32), fp]
    return L
