"""The weight scales of groups of 128 that the few-row kernels copy: for every row, K range and run of steps, the copied words hold
all of the run's pairs and no byte outside the tensor is read."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
#define __host__
#define __device__
#include "scale_words.cuh"
extern "C" int words(long long first, int n) { return amx::pair_words(first, n); }
extern "C" int whole(long long word, long long pairs) { return amx::pair_word_whole(word, pairs); }
"""


@pytest.fixture(scope="module")
def header(tmp_path_factory):
    d = tmp_path_factory.mktemp("scale_words")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2411_09909_b200", "csrc"),
                           str(d / "p.cpp"), "-o", str(d / "p.so")])
    lib = ctypes.CDLL(str(d / "p.so"))
    lib.words.argtypes, lib.whole.argtypes = (ctypes.c_longlong, ctypes.c_int), (ctypes.c_longlong, ctypes.c_longlong)
    return lib


@pytest.mark.parametrize("rows", [1, 2, 3])
@pytest.mark.parametrize("steps", [4, 5, 8, 9, 31, 32, 33, 35])
@pytest.mark.parametrize("ranges", [1, 2, 3, 8])
def test_runs_stay_inside_the_tensor(header, rows, steps, ranges):
    pairs = rows * steps
    for r in range(rows):
        for i in range(ranges):
            begin, end = steps * i // ranges, steps * (i + 1) // ranges
            for held in (4, 32):                                  # steps whose scales are held at a time: streaming, 128 rows per CTA
                for warps in (1, 8):                              # a warp's steps of a range: streaming kernel
                    for w in range(warps):
                        lo, hi = begin + (end - begin) * w // warps, begin + (end - begin) * (w + 1) // warps
                        for first in range(lo, hi, held):
                            n = min(hi - first, held)
                            start = r * steps + first
                            count = header.words(start, n)
                            assert count <= n // 2 + 1            # the room a row has in shared memory
                            read = set()
                            for word in range(start // 2, start // 2 + count):
                                if header.whole(word, pairs):
                                    read.update(range(4 * word, 4 * word + 4))
                            if pairs % 2 and r == rows - 1 and first + n == steps:   # the half word that is loaded by itself
                                assert 0 <= pairs // 2 - (pairs - n) // 2 < count
                                read.update(range(2 * pairs - 2, 2 * pairs))
                            assert max(read) < 2 * pairs
                            assert read >= set(range(2 * start, 2 * (start + n)))
