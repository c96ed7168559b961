"""What the binding takes as a stream: an integer handle. Anything else is refused before it
can reach the library as a pointer. No GPU."""
import ctypes as C
import enum

import pytest

from paper_1811_08488_gb300 import dwf


class Handle:
    _as_parameter_ = C.c_void_p(1)


@pytest.mark.parametrize("bad", ["stream", b"stream", Handle(), C.c_void_p(1), 1.0, [0]])
def test_refused(bad):
    with pytest.raises(TypeError):
        dwf._stream(bad)


def test_taken():
    assert dwf._stream(0) == 0 and dwf._stream(1 << 40) == 1 << 40
    assert dwf._stream(enum.IntEnum("E", {"A": 7}).A).value == 7
