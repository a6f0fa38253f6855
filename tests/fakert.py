"""The library's host code on a CUDA runtime without a GPU (tests/fake_cudart.cpp)."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2608_17616_gb300 import build as mbuild

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    def __init__(self, path):
        self.path = path
        self.raw = ctypes.CDLL(path)
        self.raw.fake_log.restype = ctypes.c_char_p

    def device(self, d):
        self.raw.fake_set_device(d)

    def fail_opt_ins(self, n):
        self.raw.fake_fail_opt_ins(n)

    def drain(self):
        """The log since the last call: launches as dicts, tensor maps as (base, [(dim, stride, box), ..]) each time their
        address is set; self.encoded counts the encodings."""
        launches, maps, self.encoded = [], [], 0
        for line in self.raw.fake_log().decode().splitlines():
            f = line.split()
            if f[0] == "launch":
                launches.append(dict(dev=int(f[1]), name=f[2], grid=tuple(map(int, f[3:6])), block=int(f[6]),
                                     smem=int(f[7]), cluster=int(f[8]), pdl=int(f[9])))
            elif f[0] == "encode":
                self.encoded += 1
            else:
                maps.append((int(f[1]), [tuple(map(int, p.split(":"))) for p in f[2:]]))
        self.raw.fake_clear()
        return launches, maps


def build_fake(tmp):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    mbuild.build()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(mbuild.nvcc()))), "include")
    out = os.path.join(str(tmp), "libmone_fakert.so")
    objs = [os.path.join(mbuild.BUILD, s.replace(".cu", ".o")) for s in mbuild.SOURCES]
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, os.path.join(HERE, "fake_cudart.cpp"),
                    *objs, "-o", out, "-lpthread"], check=True)
    return out
