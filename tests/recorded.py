"""The library on a runtime that runs nothing and records the kernels that are launched (fake_cudart.cpp): what the host code
does, without a GPU."""
import ctypes as C
import os
import subprocess

from paper_2405_17873_b200 import build, mixdq

HERE = os.path.dirname(os.path.abspath(__file__))
BUFFER = C.c_void_p(0x100000)  # any tensor's address: never dereferenced


def link(path: str) -> str:
    """The library's own object files, linked with that runtime."""
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I/usr/local/cuda/include",
                    os.path.join(HERE, "fake_cudart.cpp")] + build.objects() + ["-Wl,-Bsymbolic", "-o", path], check=True)
    return path


class Recorded:
    def __init__(self, path: str):
        self.so = C.CDLL(path)
        for name, (res, args) in mixdq._SIGNATURES.items():
            getattr(self.so, name).restype, getattr(self.so, name).argtypes = res, args
        self.so.fake_kernel.restype = C.c_char_p
        self.so.fake_capturing.argtypes = [C.c_void_p, C.c_int]

    def launches(self):
        """(kernel, launched with programmatic overlap) of every launch since the last call."""
        got = [(self.so.fake_kernel(i).decode(), bool(self.so.fake_overlap(i))) for i in range(self.so.fake_launches())]
        self.so.fake_clear()
        return got
