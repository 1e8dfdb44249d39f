// Pieces shared by the kernels of the 4-bit group-quantised format (Sec. 4.1, 4.4, 5.1): the packed
// layout's chunk size, the nibble-to-float16 operand trick, and small PTX wrappers.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "tetra_device.cuh"

namespace tetra {
namespace {

// Packed layout.  Rows are taken in strips of 32, columns in groups of G; the data of (strip, group) is one
// contiguous chunk of CH = (G / 64) * 1024 + 128 bytes at (strip * groups + group) * CH:
//   for each 64-column tile j of the group, two 512-byte sub-tiles h = 0, 1 (rows 16 h .. 16 h + 15 of the
//   strip) at j * 1024 + h * 512, in which lane = 4 g + t of a warp owns 16 bytes = four words m = 0..3; word m
//   holds, as nibbles n0..n7 (n_i at bits 4 i), the weights of columns c = 64 j + 16 t + 4 m + {0,1,2,3}:
//       n0, n4 = row g,     c + 0, c + 1        n1, n5 = row g,     c + 2, c + 3
//       n2, n6 = row g + 8, c + 0, c + 1        n3, n7 = row g + 8, c + 2, c + 3      (rows within the sub-tile)
//   then 32 (scale, offset) float16 pairs, one per row of the strip.
// A warp streams whole chunks; nothing else of the matrix is read.
__host__ __device__ constexpr int q4_chunk_bytes(int G) { return (G / 64) * 1024 + 128; }

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// What the lanes of a B column that carries no vector read as activations: 16 halves of each tile of a group.
constexpr int kQ4TileZeros = 192;
__device__ const uint4 q4_zeros[kQ4TileZeros / 16] = {};

// A lane's activations of a group's TILES 64-column tiles, through L1.  Global loads and cp.async are served in order: a
// load behind a copy waits for the copy's memory, so these go out before the group's copies.
template <int TILES>
__device__ __forceinline__ void load_group(const unsigned char* x, uint32_t (&xr)[TILES][8]) {
#pragma unroll
    for (int j = 0; j < TILES; ++j) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(x) + 8 * j), b = __ldg(reinterpret_cast<const uint4*>(x) + 8 * j + 1);
        xr[j][0] = a.x; xr[j][1] = a.y; xr[j][2] = a.z; xr[j][3] = a.w;
        xr[j][4] = b.x; xr[j][5] = b.y; xr[j][6] = b.z; xr[j][7] = b.w;
    }
}

// (a, a) * (b0, b1) + (c0, c1) in one instruction (fma.rn.f32x2).
__device__ __forceinline__ void fma2(float a, float b0, float b1, float& c0, float& c1) {
    uint64_t aa, bb, cc;
    asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a));
    asm("mov.b64 %0, {%1, %2};" : "=l"(bb) : "f"(b0), "f"(b1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(cc) : "f"(c0), "f"(c1));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(cc) : "l"(aa), "l"(bb));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c0), "=f"(c1) : "l"(cc));
}

__device__ __forceinline__ uint32_t lop_and_or(uint32_t a, uint32_t mask, uint32_t magic) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(mask), "r"(magic));  // (a & mask) | magic
    return r;
}
__device__ __forceinline__ void q4_lds128(uint32_t saddr, uint32_t (&v)[4]) {
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(saddr));
}
__device__ __forceinline__ void q4_cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
template <int PENDING>
__device__ __forceinline__ void q4_cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// First MMA of a group: the accumulator starts from c (minus the group's bias sums).
__device__ __forceinline__ void mma_f16_first(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, float c_even,
                                              float c_odd) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c_even), "f"(c_odd));
}


// ---------------------------------------------------------------------------
// One vector in whole numbers.  x 2^28 is an integer below 2^44 for every finite float16, six signed digits to the base
// 256, and the digits are the columns of an int8 MMA's B: column v of D is the exact sum of q times digit v over a group, a
// float without rounding (below 2^22).  The nibbles are bytes as they stand, those in the upper halves 16 times too
// large: their columns hold the digits of x 2^24.
// ---------------------------------------------------------------------------
constexpr int kQ4Digits = 6;
// Bytes from one digit's activations to the next's: two digits' reads fall into different banks.
__host__ __device__ constexpr uint32_t q4_digit_stride(int K) { return ((uint32_t(K) + 127u) & ~127u) + 64u; }
// Column v's weight; column 7 carries offset times the group's sum, column 6 nothing.
__device__ __forceinline__ float digit_weight(int v) { return v == 7 ? 1.f : __int_as_float((127 - 28 + 8 * v) << 23); }

// Digits of a float16 times 2^(24 + SHIFT): digits 0..3 and 4, 5 (two bytes above them unused).
template <int SHIFT>
__device__ __forceinline__ uint2 half_digits(uint32_t h) {
    const uint32_t e = (h >> 10) & 31u, m = (h & 0x3FFu) | (e ? 0x400u : 0u);
    const int64_t mag = int64_t(m) << (max(e, 1u) - 1u + SHIFT);
    const uint64_t q = uint64_t((h & 0x8000u) ? -mag : mag) + 0x808080808080ull;  // every digit moved up by 128
    return make_uint2(uint32_t(q) ^ 0x80808080u, uint32_t(q >> 32) ^ 0x80808080u);
}
// Eight activations: their digits go to `at` + stride * digit, in the byte order in which the weights' nibbles come.
__device__ __forceinline__ void store_digits(const uint4& u, unsigned char* at, uint32_t stride) {
    // low nibbles: columns 0, 1, 4, 5; upper ones: 2, 3, 6, 7
    const uint32_t lo[4] = {u.x & 0xFFFFu, u.x >> 16, u.z & 0xFFFFu, u.z >> 16};
    const uint32_t up[4] = {u.y & 0xFFFFu, u.y >> 16, u.w & 0xFFFFu, u.w >> 16};
    uint32_t out[2][kQ4Digits];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        uint2 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = s == 0 ? half_digits<4>(lo[i]) : half_digits<0>(up[i]);
        const uint32_t a = prmt(q[0].x, q[1].x, 0x5140u), b = prmt(q[2].x, q[3].x, 0x5140u);  // digits 0, 0, 1, 1
        const uint32_t c = prmt(q[0].x, q[1].x, 0x7362u), d = prmt(q[2].x, q[3].x, 0x7362u);  // digits 2, 2, 3, 3
        const uint32_t e = prmt(q[0].y, q[1].y, 0x5140u), f = prmt(q[2].y, q[3].y, 0x5140u);  // digits 4, 4, 5, 5
        out[s][0] = prmt(a, b, 0x5410u); out[s][1] = prmt(a, b, 0x7632u);
        out[s][2] = prmt(c, d, 0x5410u); out[s][3] = prmt(c, d, 0x7632u);
        out[s][4] = prmt(e, f, 0x5410u); out[s][5] = prmt(e, f, 0x7632u);
    }
#pragma unroll
    for (int v = 0; v < kQ4Digits; ++v) *reinterpret_cast<uint2*>(at + v * stride) = make_uint2(out[0][v], out[1][v]);
}
// NaN for an infinite or NaN sum: the digits of such an activation mean nothing, and this reaches every row.
__device__ __forceinline__ float nan_unless_finite(float v) {
    return (__float_as_uint(v) & 0x7F800000u) == 0x7F800000u ? __uint_as_float(0x7FC00000u) : v;
}
__device__ __forceinline__ void mma_digits(int (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, bool first) {
    if (first)
        asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                     : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "r"(0));
    else
        asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                     : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// D of one chunk, TILES tiles of 32 rows x 64 columns: `slot` this lane's 16 bytes of the chunk, `xd` of the digits.
template <int TILES>
__device__ __forceinline__ void digit_sums(uint32_t slot, uint32_t xd, float (&d)[2][4]) {
    int di[2][4];
#pragma unroll
    for (int j = 0; j < TILES; ++j) {
        uint32_t x[4];
        q4_lds128(xd + 64 * j, x);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t w[4];
            q4_lds128(slot + j * 1024 + h * 512, w);
#pragma unroll
            for (int m = 0; m < 4; m += 2) {
                const uint32_t r0 = prmt(w[m], w[m + 1], 0x6420u), r1 = prmt(w[m], w[m + 1], 0x7531u);  // rows g, g + 8
                const uint32_t a[4] = {r0 & 0x0F0F0F0Fu, r1 & 0x0F0F0F0Fu, r0 & 0xF0F0F0F0u, r1 & 0xF0F0F0F0u};
                mma_digits(di[h], a, x[m], x[m + 1], j == 0 && m == 0);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) d[h][i] = float(di[h][i]);
}

}  // namespace
}  // namespace tetra
