"""tc_api.cu compiled as host code against the CUDA runtime of fake_cuda.cpp."""
from __future__ import annotations

import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_2202_13976_gb300", "csrc")


def load(build_dir: str) -> ctypes.CDLL:
    from paper_2202_13976_gb300._build import nvcc
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    lib = os.path.join(build_dir, "libtc_fake.so")
    cmd = ["g++", "-std=c++17", "-O1", "-g", "-shared", "-fPIC", "-w", "-I", include, "-I", CSRC, "-x", "c++",
           os.path.join(CSRC, "tc_api.cu"), os.path.join(HERE, "fake_cuda.cpp"), "-o", lib,
           "-Wl,-Bsymbolic", "-Wl,-z,defs", "-pthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed:\n{r.stderr}")
    so = ctypes.CDLL(lib)
    P, i32, i64 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
    so.tc_graph_create_from_edges.argtypes = [i32, i64, P, P, i32, P, P]
    so.tc_batch_create.argtypes = [i32, P, P, P, P, i32, P, P]
    so.fake_undirected_rows.argtypes = [i32, i64, P, P, i32]
    so.fake_busy.argtypes = [ctypes.c_long, i32]
    so.fake_fail.argtypes = [ctypes.c_char_p, i32]
    so.fake_plan_side.restype = ctypes.c_long
    so.fake_bytes.restype = so.fake_peak.restype = ctypes.c_size_t
    return so
