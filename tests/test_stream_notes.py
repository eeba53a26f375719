"""The order of packing calls and the layer calls behind them, seen in how their kernels are launched.

A layer kernel loads its weights before it waits for earlier kernels of its stream, so the first one behind a packing call
must not be launched with programmatic overlap, unless an empty kernel stands between the two.  On the recording runtime
(recorded.py): nothing here runs on a GPU."""
import threading

import pytest

from recorded import BUFFER, Recorded

LEGACY, PER_THREAD = 1, 2


class Lib(Recorded):
    def pack(self, stream=0):
        assert self.so.mixdq_pack_weights(BUFFER, 64, 128, 8, BUFFER, None, 1, BUFFER, stream) == 0

    def layer(self, stream=0):
        return self.so.mixdq_linear_q8(BUFFER, 64, 128, BUFFER, 64, 8, BUFFER, BUFFER, None, BUFFER, None, stream)

    def launches(self):
        kind = lambda name: "empty" if "constants_complete_kernel" in name else "pack" if "pack_kernel" in name else "layer"
        return [(kind(name), overlap) for name, overlap in super().launches()]


@pytest.fixture
def lib(recorded_library):
    lib = Lib(recorded_library)
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
