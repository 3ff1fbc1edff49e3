"""The word in which a clustering round's blocks exchange their counts holds those of the largest scene that a build
accepts (2^31 - 1 triangles): fields that carried into each other would put nodes and clusters at wrong places.  The
header the kernel uses is compiled for the host."""
import ctypes
import itertools
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_10295_gb300", "csrc")
TOP = 2**31 - 1
SHIM = """
#include "ploc_counts.h"
using namespace lidar;
typedef unsigned long long u64;
extern "C" u64 counts(unsigned m, unsigned s) { return ploc_counts(m, s); }
extern "C" unsigned merges(u64 c) { return ploc_merges(c); }
extern "C" unsigned stays(u64 c) { return ploc_stays(c); }
extern "C" u64 tagged(u64 c, unsigned r) { return ploc_tagged(c, r); }
extern "C" int is_of(u64 w, unsigned r) { return ploc_is_of(w, r); }
extern "C" u64 untagged(u64 w) { return ploc_untagged(w); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("counts")
    (d / "shim.cc").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Wextra", "-Werror", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "shim.cc"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    for name, res, args in (("counts", ctypes.c_uint64, [ctypes.c_uint32] * 2), ("merges", ctypes.c_uint32, [ctypes.c_uint64]),
                            ("stays", ctypes.c_uint32, [ctypes.c_uint64]),
                            ("tagged", ctypes.c_uint64, [ctypes.c_uint64, ctypes.c_uint32]),
                            ("is_of", ctypes.c_int, [ctypes.c_uint64, ctypes.c_uint32]),
                            ("untagged", ctypes.c_uint64, [ctypes.c_uint64])):
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


EDGES = (0, 1, 2**28 - 1, 2**28, 2**28 + 1, 2**30, TOP)


@pytest.mark.parametrize("merges,stays", list(itertools.product(EDGES, EDGES)))
def test_counts_pass_whole(lib, merges, stays):
    for rnd in (0, 1, 2, 199, 200, 2**32 - 1):
        word = lib.tagged(lib.counts(merges, stays), rnd)
        assert lib.is_of(word, rnd)
        assert (lib.merges(lib.untagged(word)), lib.stays(lib.untagged(word))) == (merges, stays)
        # an empty sector and the answers of the rounds beside are not taken for this one
        assert not lib.is_of(0, rnd)
        if rnd + 1 < 2**32:
            assert not lib.is_of(lib.tagged(lib.counts(merges, stays), rnd + 1), rnd)


@pytest.mark.parametrize("n", [2**28 - 1, 2**28, 2**28 + 2**27, TOP])
@pytest.mark.parametrize("pairs", [0.0, 0.1, 0.5])
def test_sums_over_blocks(lib, n, pairs):
    """Sums of 512 blocks' words are the words of the sums."""
    merges = int(n * pairs)
    stays = n - merges
    blocks = [(merges // 512 + (b < merges % 512), stays // 512 + (b < stays % 512)) for b in range(512)]
    word = sum(lib.counts(m, s) for m, s in blocks)
    assert word < 2**62
    assert (lib.merges(word), lib.stays(word)) == (merges, stays)
