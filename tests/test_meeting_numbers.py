"""The numbers that stamp the resident kernel's meetings, over many launches of
every size (csrc/meeting_numbers.hpp, compiled for the host)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """#include "meeting_numbers.hpp"
extern "C" int take(uint32_t* last, uint32_t count, uint32_t* seq0) {
    return lpgb::take_meeting_numbers(*last, count, seq0);
}
"""


@pytest.fixture(scope="module")
def take(tmp_path_factory):
    d = tmp_path_factory.mktemp("numbers")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1803_04378_gb300", "csrc"),
                    "-o", str(d / "t.so"), str(d / "t.cpp")], check=True)
    return ctypes.CDLL(str(d / "t.so")).take


@pytest.mark.parametrize("count", [11, 326, 20486])  # launches of 2, 65 and 4097 steps
def test_numbers_until_they_begin_again(take, count):
    top = 2 ** 32
    last, seq0 = ctypes.c_uint32(top - 1 - 3 * count), ctypes.c_uint32()
    given = last.value
    for launch in range(8):
        restart = take(ctypes.byref(last), count, ctypes.byref(seq0))
        # the last number of all, 2^32 - 1, is the third launch's; the fourth begins again
        assert bool(restart) == (launch == 3)
        assert seq0.value == (0 if restart else given)
        given = seq0.value + count
        assert last.value == given < top  # no number wraps inside a launch, and 0 is never one
