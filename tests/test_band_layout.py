"""The banded scratch across calls of different sizes, from the layout's own
header compiled on the host.

A call's geometry kernel clears the query counts (qhist) while the previous
call's last kernel may still run, so those bytes belong to no other buffer of
any other call's layout."""
import ctypes
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_18401_gb300", "csrc")
FIELDS = ["qperm", "descA", "descB", "qbkt", "qsrt", "qscale", "rnorm", "fcand", "fmask", "qrank", "qhist", "part",
          "part_n", "arrived", "total"]


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src, lib = d / "layout.cpp", d / "liblayout.so"
    src.write_text('#include "band_layout.h"\n'
                   'extern "C" void layout(int64_t nq, int64_t nr, int npairs, int packed, int64_t *out) {\n'
                   "    const egm::BandLayout l(nq, nr, npairs, packed != 0);\n"
                   "    const size_t v[] = {" + ", ".join("l." + f for f in FIELDS) + "};\n"
                   f"    for (int k = 0; k < {len(FIELDS)}; k++) out[k] = (int64_t)v[k];\n"
                   "}\n")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).layout
    fn.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int64)]

    def ranges(nq, nr, npairs, packed):
        """{buffer: (first byte, one past its last)}"""
        out = (ctypes.c_int64 * len(FIELDS))()
        fn(nq, nr, npairs, int(packed), out)
        at = dict(zip(FIELDS, out))
        starts = sorted(at.values())
        return {f: (b, starts[starts.index(b) + 1]) for f, b in at.items() if f != "total"}

    return ranges


SIZES = [(1, 1), (100, 5000), (8000, 8000), (10000, 10000), (13000, 20000), (30000, 30000), (45000, 45000),
         (50000, 49999), (65000, 65000), (200000, 1000)]
CALLS = [(m, n, p, f) for m, n in SIZES for p in (1, 2, 17) for f in (False, True)]


def test_query_counts_lie_apart_from_every_buffer_of_another_call(layout):
    table = {c: layout(*c) for c in CALLS}
    for prev, call in itertools.product(CALLS, CALLS):
        lo, hi = table[call]["qhist"]
        assert hi - lo >= 4 * 2050 * min(call[2], 16)
        for name, (a, b) in table[prev].items():
            if name != "qhist":
                assert b <= lo or hi <= a, (prev, call, name)


def test_buffers_of_one_call_do_not_overlap(layout):
    for c in CALLS:
        r = sorted(layout(*c).values())
        assert all(x[1] <= y[0] for x, y in zip(r, r[1:]))
