"""Rows of activations that are not 16-byte aligned (csrc/tetra_rows.h, tetra_batched.cu): every copy of every lane, walked
through on the host.  A read ahead of the caller's activations faults nowhere and changes no result, so only the addresses
show it."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_35465_b200", "csrc")

# argv: batch, K, Kx (what the blocks cover), x's address in halves; prints what went wrong first, or nothing
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "tetra_rows.h"
using namespace tetra;
int main(int, char** argv) {
    const int V = std::atoi(argv[1]), K = std::atoi(argv[2]), Kx = std::atoi(argv[3]);
    const uint32_t x_half = uint32_t(std::atoi(argv[4]));
    const int quads = (Kx + 95) / 96;
    for (int quad = 0; quad < quads; ++quad) {
        std::vector<long> buffer(size_t(V) * 8 * kRowUnits, -1);  // what lies where: -1 nothing, -2 a zero, else half of x
        const bool begin = quad == 0 && rows_begin_within_a_unit(x_half);
        for (int v = 0; v < V; ++v) {
            const int skip = int(row_skip(x_half, v, K));
            for (int u = begin ? 1 : 0; u < kRowUnits; ++u) {
                const RowUnit unit = row_unit(uint32_t(skip), quad, u, Kx);
                const long at = long(v) * K + unit.from;
                if (unit.halves && ((long(x_half) + at) & 7)) return std::printf("vector %d quad %d unit %d: not aligned", v, quad, u), 0;
                for (int i = 0; i < 8; ++i) {
                    if (i < unit.halves && (at + i < 0 || at + i >= long(V) * K))
                        return std::printf("vector %d quad %d unit %d reads half %ld of %ld", v, quad, u, at + i, long(V) * K), 0;
                    buffer[size_t(v) * 8 * kRowUnits + 8 * u + i] = i < unit.halves ? at + i : -2;
                }
            }
            if (begin)
                for (int h = skip; h < 8; ++h) buffer[size_t(v) * 8 * kRowUnits + h] = h - skip < Kx ? long(v) * K + h - skip : -2;
            for (int j = 0; j < 96; ++j) {  // what the products read
                const int k = 96 * quad + j;
                if (buffer[size_t(v) * 8 * kRowUnits + skip + j] != (k < Kx ? long(v) * K + k : -2))
                    return std::printf("vector %d half %d is not in its place", v, k), 0;
            }
        }
    }
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "walk.cpp").write_text(PROGRAM)
    exe = str(d / "walk")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-I", CSRC, str(d / "walk.cpp"), "-o", exe], check=True)
    return lambda *a: subprocess.run([exe] + [str(v) for v in a], check=True, capture_output=True, text=True).stdout


# Rows shorter than a unit (several begin in the first one), of a few units, of several quads and not a whole last one; the
# blocks cover the row (zero-pad rule) or leave a tail.
@pytest.mark.parametrize("K,Kx", [(1, 1), (2, 2), (3, 3), (5, 5), (7, 7), (9, 9), (24, 24), (25, 24), (95, 72), (97, 97), (100, 96),
                                  (217, 216), (1685, 1680)])
@pytest.mark.parametrize("batch", [2, 3, 16])
def test_rows_are_copied_whole_and_nothing_outside_them(walk, batch, K, Kx):
    for x_half in range(8):
        assert walk(batch, K, Kx, x_half) == "", "x %d halves into a unit" % x_half


def test_the_walk_sees_a_unit_that_begins_ahead_of_x(walk, tmp_path):
    """The rule as it would be without the exception."""
    text = open(os.path.join(CSRC, "tetra_rows.h")).read()
    head = text.replace("return (x_half & 7u) != 0;", "return false;")
    assert head != text
    (tmp_path / "tetra_rows.h").write_text(head)
    (tmp_path / "walk.cpp").write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-I", str(tmp_path), str(tmp_path / "walk.cpp"), "-o", str(tmp_path / "w")], check=True)
    out = subprocess.run([str(tmp_path / "w"), "2", "25", "24", "3"], check=True, capture_output=True, text=True).stdout
    assert out.startswith("vector 0 quad 0 unit 0 reads half -3")
