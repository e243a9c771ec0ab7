"""The library's host code on a machine without a GPU: its objects linked against a CUDA runtime
that records launches instead of making them (fake_cudart.c)."""
import ctypes
import os
import re
import subprocess

from paper_2411_10948_gb300 import build, native

HERE = os.path.dirname(os.path.abspath(__file__))


def link(folder):
    """The library over the fake runtime, as native.load() gives it, with the fake's controls."""
    objs = [os.path.join(build.BUILD, f.replace(".cu", ".o")) for f in build.SOURCES]
    build.build_library()
    if not all(map(os.path.exists, objs)):
        build.build_library(force=True)
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    so = os.path.join(str(folder), "libshiftquant_fake.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-I", inc, "-o", so,
                           os.path.join(HERE, "fake_cudart.c"), *objs, "-lstdc++",
                           "-Wl,-Bsymbolic", "-Wl,--no-undefined"])
    lib = native.load(so)
    lib.fake_log.restype = ctypes.c_char_p
    return lib


def launches(lib):
    """(kernel, blocks, flags) of every launch since the last call, memsets left out."""
    out = []
    for line in lib.fake_log().decode().splitlines():
        name, n, flags = line.split()
        if name not in ("memset", "memcpy"):
            m = re.match(r"_ZN2sq(\d+)(\w+)", name)   # namespace sq, the name's length, the name
            out.append((m.group(2)[:int(m.group(1))], int(n), flags))
    return out
