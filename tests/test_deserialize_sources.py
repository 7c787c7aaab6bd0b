"""What Matrix.deserialize() reads from: any buffer, in place or copied (CPU)."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3, workloads as wl


@pytest.mark.parametrize("source", [bytes, bytearray, lambda b: memoryview(bytearray(b)), lambda b: np.frombuffer(b, dtype=np.uint8).copy(),
                                    lambda b: type("B", (bytes,), {})(b)])
def test_every_kind_of_buffer(source):
    build.build_library()
    W = wl.Case(0, "d", 130, 260, 8, 4, 0.5, "magnitude").make_W()
    m = tl3.encode(W)
    for data in (m.serialize(), m.serialize(compact=True)):
        again = tl3.Matrix.deserialize(source(data))
        assert again.serialize() == m.serialize()
        assert np.array_equal(again.decode(), m.decode())


@pytest.mark.parametrize("data", [b"", bytearray(), b"\0", bytes(200), bytearray(200), np.zeros(0, dtype=np.uint8)])
def test_what_is_no_container_is_refused(data):
    build.build_library()
    with pytest.raises(tl3.Tl3Error):
        tl3.Matrix.deserialize(data)
