"""Places of the fused loops' packets (csrc/looplayout.h), on the host.

Exchange numbers are per mesh, so what a mesh of a batch writes in any of its solves (three components
per row, one to three right-hand sides; three or one value per piece and aggregate) must stay out of
every other mesh's range, and within a solve no two values may share a place.
"""
import ctypes as C
import itertools
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2510_09812_gb300", "csrc")
SRC = """
#include "looplayout.h"
extern "C" long p3(long j, long c) { return gspm::p_packet3(j, (int)c); }
extern "C" long q1(long j) { return gspm::p_packet1((int)j); }
extern "C" long p1(long j, long c) { return gspm::p_packet1((int)j, (int)c); }
extern "C" long co(long f, long i, long nc, long c) {
  return gspm::coarse_packet((int)f, (int)i, (int)nc, (int)c);
}
"""


@pytest.fixture(scope="module")
def lay(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("layout")
    (d / "l.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "l.so"),
                    str(d / "l.cpp")], check=True)
    lib = C.CDLL(str(d / "l.so"))
    for f, n in (("p3", 2), ("q1", 1), ("p1", 2), ("co", 4)):
        getattr(lib, f).restype = C.c_long
        getattr(lib, f).argtypes = [C.c_long] * n
    return lib


def _solves(lay, first, count, rows):
    """Every solve's places of one mesh: a list per solve."""
    items = range(first, first + count)
    if rows:
        yield [lay.p3(j, c) for j in items for c in range(3)]
        for nr in (2, 3):
            yield [lay.p1(j, c) for j in items for c in range(nr)]
        # one right-hand side: an array of its own
        yield [-1 - lay.q1(j) for j in items]
    else:
        for nc in (3, 1):
            yield [lay.co(first, i, nc, c) for i in items for c in range(nc)]


@pytest.mark.parametrize("rows", [True, False])
@pytest.mark.parametrize("counts", [(32, 32), (64, 32, 160, 32), (32, 1024, 96)])
def test_ranges_of_meshes_are_disjoint(lay, counts, rows):
    if not rows:
        counts = [c // 32 for c in counts]              # pieces, aggregates: any count
    starts = [0] + list(itertools.accumulate(counts))
    used = []
    for first, count in zip(starts, counts):
        places = set()
        for solve in _solves(lay, first, count, rows):
            assert len(set(solve)) == len(solve)
            places.update(solve)
        assert min(places) >= -sum(counts) and max(places) < 3 * sum(counts)
        used.append(places)
    for a, b in itertools.combinations(used, 2):
        assert not a & b
