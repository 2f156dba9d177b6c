"""The frame descriptors of the batch calls: one struct call a frame gives the
bytes of the ctypes structures, also for values that struct refuses and ctypes
converts, and for intrinsics that can be read only once."""
import ctypes

import pytest

from paper_1707_00385_gb300 import pcurv


class Buffer:
    """What the descriptors read of a tensor."""

    def __init__(self, ptr, *shape):
        self.ptr, self.shape = ptr, shape

    def data_ptr(self):
        return self.ptr


INTRINSICS = [(525.0, 525.0, 319.5, 239.5), (525, 524, 1, -2), (1e39, -1e39, 0.0, 1.0), (float("inf"), 1.0, float("nan"), 0.5),
              ("525", 525.0, "31.5", 0.1), (True, 2.0 ** -130, 1e-46, 3.0)]
SHAPES = [(480, 640), (0, 7), (1, 1), (2 ** 31 + 5, 3)]


def test_sizes():
    assert pcurv._FRAME.size == ctypes.sizeof(pcurv.pc_frame)
    assert pcurv._PACKED_FRAME.size == ctypes.sizeof(pcurv.pc_packed_frame)


@pytest.mark.parametrize("once", [False, True])
def test_bytes_of_the_structures(once):
    read = iter if once else tuple
    frames, packed, want, want_packed = [], [], [], []
    for k, intr in enumerate(INTRINSICS):
        for m, (H, W) in enumerate(SHAPES):
            p = 2 ** 40 + 4096 * (len(SHAPES) * k + m)
            normal = None if m % 2 else Buffer(p + 768)
            out = (Buffer(p + 256), Buffer(p + 512), normal)
            ptrs = (p + 256, p + 512, normal and normal.ptr)
            frames.append((Buffer(p, H, W), read(intr), *out))
            want.append(pcurv.pc_frame(p, H, W, *map(float, intr), *ptrs))
            packed.append((Buffer(p, H, W), Buffer(p + 128), read(intr), *out))
            want_packed.append(pcurv.pc_packed_frame(p, p + 128, H, W, *map(float, intr), *ptrs))
    for got, ref in ((pcurv._frame_array(frames), want), (pcurv._packed_frame_array(packed), want_packed)):
        assert len(got) == len(ref)
        for g, w in zip(got, ref):
            assert bytes(g) == bytes(w)


def test_stream_of_a_torch_without_the_raw_handle(monkeypatch):
    torch = pytest.importorskip("torch")

    class Stream:
        cuda_stream = 17

    monkeypatch.setattr(torch.cuda, "current_stream", lambda: Stream)
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert pcurv._stream_handle(None) == 17
    assert pcurv._stream_handle(Stream) == 17
