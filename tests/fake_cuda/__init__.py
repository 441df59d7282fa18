"""The library's own objects linked with a stand-in for the CUDA runtime
(fake_cudart.cpp): the host side of every entry point then runs on the CPU,
and what it launches can be read back."""
from __future__ import annotations

import ctypes
import glob
import os
import subprocess
from dataclasses import dataclass

from paper_2606_27550_gb300 import build as tvbuild

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(tvbuild.nvcc()))), "include")


def build_lib(out_dir: str) -> str:
    """Links the fake library into out_dir and returns its path."""
    tvbuild.build()
    objs = [os.path.join(tvbuild.BUILD, os.path.basename(s) + ".o") for s in glob.glob(os.path.join(tvbuild.CSRC, "*.cu"))]
    if not all(os.path.exists(o) for o in objs):
        tvbuild.build(force=True)
    lib, fake = (os.path.join(str(out_dir), n) for n in ("libtreeverify_fake.so", "fake.o"))
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-I", CUDA_INCLUDE, "-c", os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", fake], check=True)
    # symbolic: the runtime that torch has loaded must not stand in for the fake one
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", lib, *objs, fake], check=True)
    return lib


@dataclass
class Launch:
    name: str  # the kernel's mangled name
    grid: tuple
    block: int
    cluster: int
    smem: int
    stream: int
    pdl: bool
    device: int


def launches(lib) -> list[Launch]:
    """The launches since the last call, in order."""
    lib.fake_launches.restype = ctypes.c_char_p
    out = []
    for line in lib.fake_launches().decode().splitlines():
        name, *x = line.split()
        x = [int(v) for v in x]
        out.append(Launch(name, tuple(x[:3]), x[3], x[4], x[5], x[6], bool(x[7]), x[8]))
    return out
