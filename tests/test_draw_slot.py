"""The places of a drawing block's records (csrc/draw_slot.h), compiled for the
host: every mask, the empty one too, has a place inside its own slot, and the
empty one's is no triangle's."""
import ctypes
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_06574_gb300", "csrc")

SOURCE = r"""
#include "draw_slot.h"
using namespace hexfc;
extern "C" int records(int chunk) { return slot_records(chunk); }
extern "C" int place(int j) { return slot_place(j); }
extern "C" int blank() { return kSlotBlank; }
extern "C" int next(uint32_t m) { return next_place(m); }
"""


def test_places_lie_in_their_slot(tmp_path):
    src, lib = tmp_path / "s.cpp", tmp_path / "s.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    s = ctypes.CDLL(str(lib))
    s.next.argtypes = [ctypes.c_uint32]
    n = s.records(32)
    assert s.next(0) == s.blank() and 0 <= s.blank() < n
    assert [s.place(j) for j in range(32)] == [k for k in range(n) if k != s.blank()]
    for j in range(32):
        for m in (1 << j, (0xFFFFFFFF << j) & 0xFFFFFFFF, (1 << j) | (1 << 31)):
            assert s.next(m) == s.place(j)
