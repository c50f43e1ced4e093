"""libsl1m's host code over a CUDA runtime and launchers that run nothing
(fake_device.cpp): builds it with the host compiler and gives the Python binding
on top of it."""
import ctypes as C
import importlib.util
import os
import subprocess
import sysconfig

from paper_1310_2078_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
HOST_SOURCES = ("sl1m_host.cpp", "sl1m_gridplan.cpp", "sl1m_server.cpp", "sl1m_refine.cpp")


def _cuda_include():
    nvcc = b._nvcc()
    root = os.path.dirname(os.path.dirname(nvcc)) if os.path.isabs(nvcc) else "/usr/local/cuda"
    for d in (os.path.join(root, "include"), os.path.join(root, "targets", "sbsa-linux", "include"),
              os.path.join(root, "targets", "x86_64-linux", "include")):
        if os.path.exists(os.path.join(d, "cuda_runtime.h")):
            return d
    raise RuntimeError(f"no CUDA headers under {root} ({sysconfig.get_platform()})")


def build(out_dir):
    """The library, in out_dir."""
    lib = os.path.join(out_dir, "libsl1m_fake.so")
    srcs = [os.path.join(b.CSRC, f) for f in HOST_SOURCES] + [os.path.join(HERE, "fake_device.cpp")]
    inc = ["-I", _cuda_include(), "-I", os.path.join(b.ROOT, "include"), "-I", b.CSRC]
    procs = []
    for s in srcs:
        o = os.path.join(out_dir, os.path.basename(s) + ".o")
        procs.append((o, subprocess.Popen(["g++", "-std=c++17", "-O1", "-g", "-fPIC", *inc, "-c", s, "-o", o])))
    for o, p in procs:
        assert p.wait() == 0, o
    # (its own cudaMalloc and the rest, whatever else the process has loaded)
    subprocess.check_call(["g++", "-shared", "-pthread", "-Wl,-Bsymbolic", "-o", lib, *(o for o, _ in procs)])
    return lib


def binding(lib):
    """A copy of the Python binding of its own that loads `lib`."""
    spec = importlib.util.spec_from_file_location("sl1m_on_fake_device", os.path.join(b.HERE, "sl1m.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    m.LIB_PATH = lib
    m.fake = m.load()
    for f, args, res in (("fake_faults", [], C.c_char_p), ("fake_reset", [], None),
                         ("fake_fail", [C.c_size_t, C.c_int], None), ("fake_total", [C.c_size_t], None), ("fake_hold", [C.c_int], None),
                         ("fake_no_threads", [C.c_int], None), ("fake_host_limit", [C.c_size_t], None),
                         ("fake_held", [], C.c_size_t), ("fake_peak", [], C.c_size_t),
                         ("fake_count", [C.c_int], C.c_longlong)):
        fn = getattr(m.fake, f)
        fn.argtypes, fn.restype = args, res
    return m
