"""Builds and loads tests/cuda/user_push_types.cu against the public device
header alone, for sm_103a."""

from __future__ import annotations

import ctypes
import os
import subprocess

from paper_2209_00103_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "cuda", "user_push_types.cu")
OUT = os.path.join(HERE, "cuda", "_build", "libgga_user_types.so")
HEADERS = [os.path.join(build.INCLUDE, f) for f in ("gga_device.cuh", "gga_layout.cuh", "gga.h")]


def build_user() -> str:
    if os.path.exists(OUT) and all(os.path.getmtime(d) <= os.path.getmtime(OUT) for d in [SRC] + HEADERS):
        return OUT
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    tmp = OUT + f".tmp{os.getpid()}"
    cmd = [build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I" + build.INCLUDE, "-Xcompiler", "-fPIC", "-shared",
           "-cudart", "shared", "-o", tmp, SRC]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
    os.replace(tmp, OUT)
    return OUT


def load_user() -> ctypes.CDLL:
    lib = ctypes.CDLL(build_user())
    vp, u32, u64, i32 = ctypes.c_void_p, ctypes.c_uint32, ctypes.c_uint64, ctypes.c_int
    lib.user_push_typed.argtypes = [vp, u32, u32, u32, u32, vp]
    lib.user_push_counted.argtypes = [vp, u32, u32, u64, i32, vp, vp, vp]
    for name in ("user_push_typed", "user_push_counted"):
        getattr(lib, name).restype = ctypes.c_int
    return lib
