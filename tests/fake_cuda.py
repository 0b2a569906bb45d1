"""Builds the library's objects against fake_cuda.cpp and loads the result: the whole C ABI with
its host logic, on a machine without a GPU."""
import ctypes as C
import os
import subprocess

from paper_2301_07264_gb300 import arso, build

HERE = os.path.dirname(os.path.abspath(__file__))


def load(tmp):
    # bound to its own symbols: another module of the process may have loaded the real runtime
    build.build()
    inc = os.path.join(build._cuda_home(), "include")
    out = os.path.join(str(tmp), "libarso_fake.so")
    objs = [os.path.join(build.OUT_DIR, f) for f in sorted(os.listdir(build.OUT_DIR)) if f.endswith(".o")]
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-I", inc, "-o", out,
                    os.path.join(HERE, "fake_cuda.cpp"), *objs, "-lpthread"], check=True)
    lib = C.CDLL(out)
    for name, args in arso._sigs.items():
        getattr(lib, name).argtypes = args
    for name in ("arso_circuit_free", "arso_error_list_free", "arso_surrogate_free"):
        getattr(lib, name).argtypes, getattr(lib, name).restype = [C.c_void_p], None
    for name in ("violation", "trims", "frees", "largest", "live", "allocs", "tried", "launches"):
        getattr(lib, "fake_" + name).restype = C.c_uint64
    lib.fake_launches.argtypes = [C.c_char_p]
    lib.fake_fail_at.argtypes = lib.fake_fail_launch_at.argtypes = [C.c_long]
    lib.fake_stream.restype = C.c_void_p
    lib.arso_last_error.restype = C.c_char_p
    return lib
