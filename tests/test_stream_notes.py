"""The order of packing calls and the layer calls behind them, seen in how their kernels are launched.

A layer kernel loads its weights before it waits for earlier kernels of its stream, so the first one behind a packing call
must not be launched with programmatic overlap, unless an empty kernel stands between the two.  The library's object files
are linked with a runtime that only records (fake_cudart.cpp): nothing here runs on a GPU."""
import ctypes as C
import os
import subprocess
import threading

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
BUFFER = C.c_void_p(0x100000)  # never dereferenced
LEGACY, PER_THREAD = 1, 2
EMPTY = "constants_complete_kernel"


@pytest.fixture(scope="session")
def fake_lib(tmp_path_factory):
    """Path of the library on the recording runtime."""
    from paper_2405_17873_b200 import build
    out = str(tmp_path_factory.mktemp("fake") / "libmixdq_fake.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I/usr/local/cuda/include", os.path.join(HERE, "fake_cudart.cpp")]
                   + build.objects() + ["-Wl,-Bsymbolic", "-o", out], check=True)
    return out


class Lib:
    def __init__(self, path):
        from paper_2405_17873_b200 import mixdq
        self.so = C.CDLL(path)
        for name, (res, args) in mixdq._SIGNATURES.items():
            if hasattr(self.so, name):
                getattr(self.so, name).restype, getattr(self.so, name).argtypes = res, args
        self.so.fake_kernel.restype = C.c_char_p
        self.so.fake_capturing.argtypes = [C.c_void_p, C.c_int]

    def pack(self, stream=0):
        assert self.so.mixdq_pack_weights(BUFFER, 64, 128, 8, BUFFER, None, 1, BUFFER, stream) == 0

    def layer(self, stream=0):
        return self.so.mixdq_linear_q8(BUFFER, 64, 128, BUFFER, 64, 8, BUFFER, BUFFER, None, BUFFER, None, stream)

    def launches(self):
        """(kernel, launched with overlap) of every launch since the last call."""
        names = [self.so.fake_kernel(i).decode() for i in range(self.so.fake_launches())]
        got = [("empty" if EMPTY in n else "pack" if "pack_kernel" in n else "layer", bool(self.so.fake_overlap(i)))
               for i, n in enumerate(names)]
        self.so.fake_clear()
        return got


@pytest.fixture
def lib(fake_lib):
    lib = Lib(fake_lib)
    for d in (1, 0):  # no note of another test stands
        lib.so.fake_device(d)
        for stream in (0, 0x70):
            lib.layer(stream)
    lib.so.fake_clear()
    return lib


@pytest.mark.parametrize("stream", [0, 0x70])
def test_first_layer_behind_a_packing_call_is_launched_plainly(lib, stream):
    lib.pack(stream)
    assert lib.layer(stream) == 0 and lib.layer(stream) == 0
    assert lib.launches() == [("pack", False), ("layer", False), ("layer", True)]


def test_default_streams_of_two_devices_are_two_streams(lib):
    for d in (0, 1):
        lib.so.fake_device(d)
        lib.pack()
    for d in (0, 1, 0, 1):
        lib.so.fake_device(d)
        assert lib.layer() == 0
    assert lib.launches() == [("pack", False)] * 2 + [("layer", False)] * 2 + [("layer", True)] * 2


def test_per_thread_stream_gets_the_empty_kernel(lib):
    """Its handle is another stream in every thread: no note is left for it."""
    lib.pack(PER_THREAD)
    thread = threading.Thread(target=lambda: lib.layer(PER_THREAD))
    thread.start()
    thread.join()
    assert lib.layer(PER_THREAD) == 0
    assert lib.launches() == [("pack", False), ("empty", False), ("layer", True), ("layer", True)]


def test_captured_launch_leaves_the_note_standing(lib):
    lib.pack(0x70)
    lib.so.fake_capturing(0x70, 1)
    assert lib.layer(0x70) == 0
    lib.so.fake_capturing(0x70, 0)
    assert lib.layer(0x70) == 0 and lib.layer(0x70) == 0
    assert lib.launches() == [("pack", False), ("layer", False), ("layer", False), ("layer", True)]


def test_captured_packing_call_ends_with_the_empty_kernel(lib):
    lib.so.fake_capturing(0x70, 1)
    lib.pack(0x70)
    assert lib.layer(0x70) == 0
    lib.so.fake_capturing(0x70, 0)
    assert lib.layer(0x70) == 0
    assert lib.launches() == [("pack", False), ("empty", False), ("layer", True), ("layer", True)]


def test_failed_launch_leaves_the_note_standing(lib):
    lib.pack()
    lib.so.fake_fail_launch()
    assert lib.layer() != 0
    assert lib.layer() == 0
    assert lib.launches() == [("pack", False), ("layer", False)]


def test_default_stream_by_its_other_handle(lib):
    lib.pack(LEGACY)
    assert lib.layer() == 0 and lib.layer(LEGACY) == 0
    assert lib.launches() == [("pack", False), ("layer", False), ("layer", True)]


def test_more_streams_than_notes(lib):
    """Beyond the notes that are kept, packing calls end with the empty kernel; every first layer stays ordered."""
    streams = range(0x1000, 0x1000 + 70 * 16, 16)
    for s in streams:
        lib.pack(s)
    assert lib.launches().count(("empty", False)) == 70 - 64
    for s in streams:
        lib.layer(s)
    assert lib.launches() == [("layer", False)] * 64 + [("layer", True)] * 6
