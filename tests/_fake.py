"""libgsis linked with a CUDA runtime that runs nothing (fake_cudart.cpp), for checks of the
host side on the CPU."""
import ctypes as C
import importlib.util
import os
import shutil
import subprocess

from paper_2601_03935_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(folder):
    """The binding module of a libgsis.so made in `folder`; the module's ``fake`` is the library."""
    build.build()
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc_path())))
    lib = os.path.join(folder, "libgsis.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + os.path.join(cuda, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", lib], check=True)
    shutil.copy(os.path.join(build.HERE, "gsis.py"), folder)
    spec = importlib.util.spec_from_file_location("gsis_without_device", os.path.join(folder, "gsis.py"))
    G = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(G)
    G.fake = G.load()
    G.fake.fake_report.restype = C.c_char_p
    G.fake.fake_launch.restype = C.c_char_p
    G.fake.fake_cleared.argtypes = [C.c_size_t]
    G.fake.fake_device_bytes.restype = C.c_size_t
    G.fake.fake_fail_malloc_after.argtypes = [C.c_longlong]
    return G


def report(G, kind=""):
    return [s for s in G.fake.fake_report().decode().split("\n") if s.startswith(kind) and s]
