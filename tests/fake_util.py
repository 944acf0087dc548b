"""The library's host code on a stand-in for the CUDA runtime (fake_cuda/): its
own objects, linked with a runtime that logs launches instead of running them."""
import ctypes
import os
import shutil
import subprocess
import threading

import paper_1808_00963_gb300 as ss

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCE = os.path.join(HERE, "fake_cuda", "fake_runtime.cpp")
BUILD = os.path.join(HERE, "fake_cuda", "_build")


def build():
    """Path of the linked library."""
    ss.build()
    os.makedirs(BUILD, exist_ok=True)
    objs = sorted(os.path.join(os.path.dirname(ss.LIB_PATH), s.replace(".cu", ".o")) for s in ss.SOURCES)
    out = os.path.join(BUILD, "libss_fake.so")
    if ss._stale(out, objs + [SOURCE]):
        include = os.path.join(os.path.dirname(os.path.dirname(ss._nvcc())), "include")
        # symbolic: a CUDA runtime that the process has loaded must not take the place of the stand-in
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-z,defs", "-Wl,-Bsymbolic", "-I", include,
                        "-o", out + ".tmp", SOURCE, *objs, "-lpthread"], check=True)
        os.replace(out + ".tmp", out)
    return out


def load(tmp_path):
    """An instance of the library of its own (loaded from a copy, so that nothing it keeps is shared)."""
    lib = ss.load(shutil.copy(build(), str(tmp_path)))
    lib.fake_log.restype = ctypes.c_size_t
    lib.fake_log.argtypes = [ctypes.c_char_p, ctypes.c_size_t]
    lib.fake_host_word.restype = ctypes.c_void_p
    lib.fake_peak.restype = ctypes.c_size_t
    lib.fake_capture.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return lib


def log(lib):
    """What was launched, in order: (thread's tag, device, stream, kernel / "graph" / "wait", first 8 bytes of the
    first parameter)."""
    size = lib.fake_log(None, 0)
    buf = ctypes.create_string_buffer(size + 1)
    lib.fake_log(buf, size + 1)
    out = []
    for line in buf.value.decode().splitlines():
        tag, device, stream, what, first = line.split(" ")
        out.append((int(tag), int(device), int(stream), what, int(first)))
    return out


def in_threads(*calls):
    """Runs the calls at the same time, each in a thread of its own; returns what they returned."""
    out = [None] * len(calls)
    gate = threading.Barrier(len(calls))

    def work(i, call):
        gate.wait()
        out[i] = call()

    threads = [threading.Thread(target=work, args=x) for x in enumerate(calls)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return out
