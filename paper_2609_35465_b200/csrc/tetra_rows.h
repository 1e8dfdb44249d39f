// Rows of activations that are not 16-byte aligned, as tetra_batched.cu brings them in: which 16 bytes a copy takes.  Plain
// C++, so that a host program can walk through every copy (tests/test_batched_rows.py).
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define TETRA_HD __host__ __device__
#else
#define TETRA_HD
#endif

namespace tetra {

// A row's share of four block columns is 96 halves.  It lies in thirteen aligned units of eight, its first half `skip`
// halves into the first of them, the same for every quad of columns (192 bytes).
constexpr int kRowUnits = 13;
// x_half: the address of the first vector, in halves.
TETRA_HD constexpr uint32_t row_skip(uint32_t x_half, int v, int K) { return (x_half + uint32_t(v) * uint32_t(K)) & 7u; }
struct RowUnit {
    int from, halves;  // halves from .. from + halves - 1 of the row; zeros for the rest of the eight
};
// Unit u of a quad; the row has Kx halves.
TETRA_HD constexpr RowUnit row_unit(uint32_t skip, int quad, int u, int Kx) {
    const int from = 96 * quad + 8 * u - int(skip), left = Kx - from;
    return {from, left < 0 ? 0 : (left > 8 ? 8 : left)};
}
// A row's first unit begins up to seven halves ahead of the row: with the end of the row before, or, for the rows that
// begin within the first vector's first unit, with memory that is not the call's.  `from` counts from the row, so the
// latter is v K + from < 0.  If x itself is aligned no unit does that; if not, the first units of quad 0 are not copied,
// their halves are loaded one by one.
TETRA_HD constexpr bool rows_begin_within_a_unit(uint32_t x_half) { return (x_half & 7u) != 0; }

}  // namespace tetra
