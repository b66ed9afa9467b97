"""The library's host code on a CUDA runtime of host memory (host_runtime.cpp):
builds it with the host compiler and returns a copy of the Python binding that
calls it. Every load is a fresh copy with its own counters and memory."""
import ctypes
import importlib.util
import os
import shutil
import subprocess
import tempfile

import paper_1311_0378_gb300 as rc
from paper_1311_0378_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


_built = []


def _build(folder):
    nvcc = shutil.which(build._nvcc()) or build._nvcc()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    lib = os.path.join(folder, "librecon_host.so")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                           "-I", inc, "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-o", lib,
                           "-x", "c++", os.path.join(HERE, "host_runtime.cpp"), os.path.join(build.CSRC, "recon_api.cu"),
                           os.path.join(build.CSRC, "recon_sched.cu")])
    return lib


def load(tmp_path):
    if not _built:
        folder = tempfile.TemporaryDirectory()   # kept, and removed at exit, with the list
        _built[:] = [_build(folder.name), folder]
    lib = shutil.copy(_built[0], str(tmp_path))
    spec = importlib.util.spec_from_file_location("recon_host", rc.__file__)
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    m.LIB_PATH = lib
    L = m.lib()
    L.ht_device_limit.argtypes = L.ht_pinned_limit.argtypes = [ctypes.c_size_t]
    L.ht_device_bytes.restype = ctypes.c_size_t
    return m


def counts(m):
    v = (ctypes.c_int * 4)()
    m.lib().ht_counts(v)
    return dict(zip(("merging", "wavefront", "graph", "plan"), v))
