// Device-side decoders for Tetra words (sm_100a).
//
// Two decoders live here:
//   * decode_file_word: the six-load decode of Sec. 3.4 (Fig. "decode") on a
//     word in file order, reading the paper-format tables.  Used by
//     tetra_decode_blocks and by the paper-design GEMV.
//   * the fast decoder: works on the re-ordered 48-bit device word written by
//     tetra_pack_codes and on tables staged in shared memory.  It produces MINUS
//     EIGHT TIMES the lattice point as packed int8, four coordinates per
//     register, with two logic operations per four (see fast_decode).
#pragma once
#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "tetra_tables.h"

namespace tetra {

// ---------------------------------------------------------------------------
// small wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
__device__ __forceinline__ int dp4a_ss(uint32_t a, uint32_t b, int c) {  // signed a . signed b
    int d;
    asm("dp4a.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int dp4a_su(uint32_t a, uint32_t b, int c) {  // signed a . unsigned b
    int d;
    asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// c + the low (HIGH: high) two bytes of b . the half words of a, all signed
template <bool HIGH>
__device__ __forceinline__ int dp2a(uint32_t a, uint32_t b, int c) {
    int d;
    if (HIGH) asm("dp2a.hi.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    else asm("dp2a.lo.s32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
// Loads from the staged tables: they never change after staging, so the loads
// are not volatile and the compiler may schedule them freely.
__device__ __forceinline__ uint32_t lds32(uint32_t saddr) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(saddr));
    return v;
}
__device__ __forceinline__ float lds32f(uint32_t saddr) {
    float v;
    asm("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(saddr));
    return v;
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  A kernel that calls pdl_release lets the next
// kernel of the stream start early; pdl_wait waits until every kernel before has
// completed and its writes are visible.  Both are no-ops for a kernel launched
// without the attribute.
//   * The products read weights (codes, row scales, tails, tables, plans) ahead of
//     pdl_wait, activations and everything else behind it.  Nothing orders a read
//     ahead of the wait behind the stores of a predecessor that has released, so a
//     kernel that writes weights (k_pack, k_q4_pack) never calls pdl_release,
//     wherever its stores are: its dependents start when it has completed.
//   * A kernel that releases also waits, all of its CTAs, so that the completion of
//     a kernel implies that of all kernels before it.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------------------
// File-order decode (Sec. 3.3, 3.4)
// ---------------------------------------------------------------------------

// The rho-th element of o + 4Z counted outward from zero, in closed form:
// v0 = 0, 4, -4, 8, -8, ... is the o = 0 list; the other lists are 1 - v0,
// 2 - v0 and v0 - 1.
__device__ __forceinline__ int rank_value(int o, int rho) {
    const int t = (rho + 1) >> 1;
    const int v0 = (rho & 1) ? 4 * t : -4 * t;
    return o == 0 ? v0 : (o == 1 ? 1 - v0 : (o == 2 ? 2 - v0 : v0 - 1));
}

__device__ __forceinline__ uint64_t load_file_word(const uint8_t* codes, size_t block) {
    const uint16_t* p = reinterpret_cast<const uint16_t*>(codes + 6 * block);
    return uint64_t(p[0]) | (uint64_t(p[1]) << 16) | (uint64_t(p[2]) << 32);
}

// T may point to global or shared memory.
__device__ __forceinline__ void decode_file_word(const PaperTables* T, uint64_t w, int y[24], int* m, int* g) {
    const int i1 = int(w & 0x7FF), i2 = int((w >> 11) & 0x7FF), i3 = int((w >> 22) & 0x7FF);
    const int s8 = int((w >> 33) & 63), b1 = int((w >> 39) & 1), b2 = int((w >> 40) & 15), b3 = int((w >> 44) & 1);
    const int p = int((w >> 45) & 1), r = int((w >> 46) & 1);
    *g = int((w >> 47) & 1);
    // trellis: the suffix read waits for the state returned by the branch read
    const int c1 = T->prefixes[2 * s8 + b1];
    const int br = T->branches[16 * s8 + b2];
    const int c3 = T->suffixes[2 * (br >> 8) + b3];
    const int c[3] = {c1, br & 0xFF, c3};
    // rank rows
    const int delta = i2 >= kMiddleClass0;
    const int r3 = p ^ r ^ delta;  // Eq. (3)
    const uint32_t row[3] = {T->rows[2048 * r + i1],
                             T->rows[delta ? 2048 + (i2 - kMiddleClass0) : i2],
                             T->rows[2048 * r3 + i3]};
    int norm = 0;
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int o = p + 2 * ((c[s] >> j) & 1);
            const int v = rank_value(o, int((row[s] >> (4 * j)) & 15u));
            y[8 * s + j] = v;
            norm += v * v;
        }
    *m = norm >> 4;
}

// ---------------------------------------------------------------------------
// Device word (written by the pack kernel).  48 bits = w0 (32) + w1 (16):
//   w0: [2..12] i1  [13] r  [14..24] i3  [25..28] a  [29] g  [30, 31, 0, 1] b
//   w1: [0..10] i2  [11] p  [12..15] x
// (a, b, x) are the Turyn coordinates of the trellis path: the three pattern
// bytes are h(a)+h'(x), h(b)+h'(x), h(a)+h(b)+h'(x).  i1 with r above it is a
// byte offset into the row table as it stands; b is one rotation away from its
// place in a table offset; p sits where i2's byte offset ends and below x, so
// that (x, p) is one five-bit index; g is in the word shifted for i3 where it
// picks the gain's table (see scale_address).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void file_to_device_word(uint64_t w, uint32_t abx, uint32_t* w0, uint32_t* w1) {
    const uint32_t i1 = uint32_t(w & 0x7FF), i2 = uint32_t((w >> 11) & 0x7FF), i3 = uint32_t((w >> 22) & 0x7FF);
    const uint32_t p = uint32_t((w >> 45) & 1), r = uint32_t((w >> 46) & 1), g = uint32_t((w >> 47) & 1);
    const uint32_t a = abx & 15u, b = (abx >> 4) & 15u, x = abx >> 8;
    *w0 = (i1 << 2) | (r << 13) | (i3 << 14) | (a << 25) | (g << 29) | (b << 30) | (b >> 2);
    *w1 = i2 | (p << 11) | (x << 12);
}
// The twelve trellis bits of a file-order word: index of DeviceTables::trellis_to_abx.
__device__ __forceinline__ uint32_t trellis_path(uint64_t w) { return uint32_t((w >> 33) & 0xFFF); }

// Byte offsets of the staged tables inside the shared-memory copy of the fast part.
constexpr uint32_t kSmRows = 0;
constexpr uint32_t kSmMid = 16384;
constexpr uint32_t kSmScale = 24576;
constexpr uint32_t kSmMaskH = 24832;
constexpr uint32_t kSmMaskXp = 24960;
constexpr uint32_t kSmGap = 25088, kStagedGap = 512;  // nothing to stage there
constexpr uint32_t kScaleGain = 1024;  // from one gain's scale table to the other's
constexpr int kNormShift = 7;          // from the squared norm of eight times the point (1024 m) to bytes of a scale table
// In a cluster a shared-memory address holds the CTA's rank from bit 24 on.  NibbleBlock::norm0 keeps an address shifted left,
// so only the rank's lowest bits are left in it: with more CTAs the lookups would go to another CTA's copy of the table (the
// same entries, through the cluster's network).
constexpr int kNormClusterMax = 1 << (32 - 24 - kNormShift);
constexpr uint32_t kSmAlign = 16384;  // the staged copy starts on a 16 KiB boundary of shared memory
static_assert(kSmMid == offsetof(DeviceTables, mid_fast) - kFastOffset, "staged layout");
static_assert(kSmScale == offsetof(DeviceTables, scale) - kFastOffset, "staged layout");
static_assert(kSmScale + kScaleGain == offsetof(DeviceTables, scale1) - kFastOffset && kSmScale % (2 * kScaleGain) == 0, "staged layout");
static_assert(sizeof(DeviceTables::scale) / 32 << kNormShift == 1024, "bytes per norm");
static_assert(kSmMaskH == offsetof(DeviceTables, mask_h) - kFastOffset && kSmMaskH % 64 == 0, "staged layout");
static_assert(kSmMaskXp == offsetof(DeviceTables, mask_xp) - kFastOffset && kSmMaskXp % 128 == 0, "staged layout");

// Copies the staged part of the tables to the first 16 KiB boundary of the
// CTA's dynamic shared memory (all threads; the caller synchronises) and returns
// that address.  The launch must reserve kFastBytes + kSmAlign bytes for it.
__device__ __forceinline__ unsigned char* stage_fast_tables(const DeviceTables* tab, unsigned char* smem) {
    const uint32_t s = smem_u32(smem);
    unsigned char* base = smem + (((s + kSmAlign - 1) & ~(kSmAlign - 1)) - s);
    const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(tab) + kFastOffset);
    uint4* dst = reinterpret_cast<uint4*>(base);
    for (uint32_t i = threadIdx.x; i < kFastBytes / 16; i += blockDim.x) dst[i] = src[i];
    return base;
}
// The same copy with cp.async (16 bytes per request, all of a thread's requests in flight at once);
// the caller commits and waits for the group and synchronises the CTA before the tables are read.
__device__ __forceinline__ unsigned char* stage_fast_tables_async(const DeviceTables* tab, unsigned char* smem) {
    const uint32_t s = smem_u32(smem);
    const uint32_t pad = ((s + kSmAlign - 1) & ~(kSmAlign - 1)) - s;
    const char* src = reinterpret_cast<const char*>(tab) + kFastOffset;
    for (uint32_t i = threadIdx.x; i < (kFastBytes - kStagedGap) / 16; i += blockDim.x) {
        const uint32_t at = 16u * i + (16u * i >= kSmGap ? kStagedGap : 0u);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(s + pad + at), "l"(src + at));
    }
    return smem + pad;
}
constexpr uint32_t kTableSmemBytes = uint32_t(kFastBytes) + kSmAlign;

struct FastBlock {
    // MINUS EIGHT TIMES the lattice point, int8 x 4: y[2 s] holds coordinates 8 s + 2, 6, 3, 7 of section s in
    // its bytes 0..3, y[2 s + 1] coordinates 8 s + 0, 4, 1, 5.  The activations' planes use the same order.
    uint32_t y[6];
    uint32_t norm0;  // what the squared norm starts from (see scale_address)
};
// Coordinate of a block held by byte i of word k.
__host__ __device__ constexpr int word_coordinate(int k, int i) { return 8 * (k >> 1) + 4 * (i & 1) + (i >> 1) + ((k & 1) ? 0 : 2); }
static_assert(fast_nibble(word_coordinate(0, 1)) == 3 && fast_nibble(word_coordinate(1, 2)) == 4 && fast_nibble(word_coordinate(0, 2)) == 5,
              "byte i of the high (low) nibbles is nibble 2 i + 1 (2 i)");

// A row table entry holds, per coordinate, the nibble -2 k, where 4 k = 0, 4, -4, 8, -8 is the rank's element of
// the o = 0 list (Sec. 3.3).  The lists of o = p + 2 c are 4 k, 1 - 4 k, 2 - 4 k, 4 k - 1, so with the nibble z
// complemented where the pattern bit c is set and once more everywhere if p = 1,
//     -y = 2 z + p     for all four lists and all five ranks
// (two's complement, -5 <= z <= 4).  The pattern masks and the complement for p are XORs; z moves to the upper
// half of its byte and p below it: a byte 16 z + 8 p = -8 y costs half a logic operation.
struct NibbleBlock {
    uint32_t z[3];  // section s: coordinate j's z at bits 4 fast_nibble(j)
    uint32_t p4;    // bit 2: p (the other bits are an address)
    uint32_t norm0; // 128 times the shared-memory address of the gain's scale table; clusters: kNormClusterMax
};
// HI = false: w1 sits in bits 0..15 of `w1pair`; HI = true: in bits 16..31.
// sm_tab: shared-memory address of the staged tables, a multiple of 16 KiB, so
// that every index is merged with its table's address by the same LOP3 that
// masks it.
template <bool HI>
__device__ __forceinline__ void decode_nibbles(uint32_t sm_tab, uint32_t w0, uint32_t w1pair, NibbleBlock& out) {
    const uint32_t sh = HI ? w1pair >> 14 : w1pair << 2;                 // [2..12] i2, [13] p, [14..17] x
    const uint32_t addr1 = (w0 & 0x3FFCu) | (sm_tab + kSmRows);          // (i1 | r << 11) * 4
    const uint32_t addr2 = (sh & 0x1FFCu) | (sm_tab + kSmMid);
    const uint32_t w3 = w0 >> 12;
    const uint32_t addr3i = (w3 & 0x1FFCu) | (sm_tab + kSmRows);
    const uint32_t a4 = ((w0 >> 23) & 0x3Cu) | (sm_tab + kSmMaskH);
    const uint32_t b4 = (__funnelshift_l(w0, w0, 4) & 0x3Cu) | (sm_tab + kSmMaskH);
    const uint32_t x4 = ((sh >> 11) & 0x7Cu) | (sm_tab + kSmMaskXp);     // (p | x << 1) * 4
    out.norm0 = (w3 & (kScaleGain << kNormShift)) | ((sm_tab + kSmScale) << kNormShift);
    const uint32_t row1 = lds32(addr1);
    const uint32_t row2 = lds32(addr2);
    // class of row 3 (Eq. (3)): p ^ r ^ delta, delta = [i2 >= 1240] = bit 11 of i2 + 808; all three at bit 13
    // (the table bases are multiples of 16 KiB, so they do not disturb bits 0..13)
    const uint32_t row3 = lds32(addr3i ^ ((addr1 ^ (addr2 + 808u * 4u) ^ sh) & 0x2000u));
    const uint32_t ma = lds32(a4);
    const uint32_t mb = lds32(b4);
    const uint32_t mx = lds32(x4);
    out.z[0] = row1 ^ ma ^ mx;
    out.z[1] = row2 ^ mb ^ mx;
    out.z[2] = row3 ^ (ma ^ mb) ^ mx;
    out.p4 = x4;
}
template <bool HI>
__device__ __forceinline__ void fast_decode(uint32_t sm_tab, uint32_t w0, uint32_t w1pair, FastBlock& out) {
    NibbleBlock nb;
    decode_nibbles<HI>(sm_tab, w0, w1pair, nb);
    out.norm0 = nb.norm0;
    const uint32_t p8 = (nb.p4 & 4u) * 0x02020202u;                      // 8 p in every byte
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        out.y[2 * s] = (nb.z[s] & 0xF0F0F0F0u) | p8;
        out.y[2 * s + 1] = ((nb.z[s] << 4) & 0xF0F0F0F0u) | p8;
    }
}

// Shared-memory address of -gain[g] / sqrt(16 m).  The squared norm of the packed point is 64 * 16 m and a gain's table
// has 8 bytes per m (16 m <= 416 for every word, Sec. 3.4), so the sum that starts from 128 times the table's address is
// 128 times the entry's; the second gain's table lies kScaleGain bytes on, which is g where the word shifted for i3 has it.
__device__ __forceinline__ uint32_t scale_address(const FastBlock& fb) {
    int n2 = int(fb.norm0);
#pragma unroll
    for (int k = 0; k < 6; ++k) n2 = dp4a_ss(fb.y[k], fb.y[k], n2);
    return uint32_t(n2) >> kNormShift;
}

// sum of -y q from the sums of -8 y over the planes of q (high signed, middle, low): every term is a multiple of
// 8 and |sum y q| <= sqrt(24 * 416) * 2^23 < 2^30, so the int32 is exact.
__device__ __forceinline__ int combine_planes(int dh, int dm, int dl) { return dh * 8192 + ((dm * 256 + dl) >> 3); }
// the same from two planes, high signed sixteen bits and low eight
__device__ __forceinline__ int combine_planes(int dh, int dl) { return dh * 32 + (dl >> 3); }

// ---------------------------------------------------------------------------
// Activations
// ---------------------------------------------------------------------------
// Fixed-point image of one block column of activations (20 words).
// step = 2^(E-22) with 2^E <= max|x| < 2^(E+1); q_j = rint(x_j / step), |q_j| < 2^23,
// stored as three byte planes (bits 23..16 signed, 15..8 and 7..0 unsigned), four
// coordinates per 32-bit word in the decoder's order (word_coordinate): words 0..5 high, 6..11 middle, 12..17 low plane;
// word 18 = step (float), word 19 is spare.  A float16 x_j is held exactly when
// |x_j| >= 2^(E-12); smaller ones are rounded to a multiple of the step.  If a value
// is NaN or infinite the step is NaN (and the planes zero).
// The 24 activations of block column c, as twelve pairs of float16 (zeros beyond K).
__device__ __forceinline__ void load_column(const __half* __restrict__ x, int K, int c, uint32_t (&w)[12]) {
    const int k0 = 24 * c;
    if (k0 + 24 <= K && ((reinterpret_cast<uintptr_t>(x) & 15) == 0)) {  // 48-byte column, 16-byte aligned
        const uint4* src = reinterpret_cast<const uint4*>(x + k0);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint4 u = __ldg(src + i);
            w[4 * i] = u.x;
            w[4 * i + 1] = u.y;
            w[4 * i + 2] = u.z;
            w[4 * i + 3] = u.w;
        }
    } else {
        const unsigned short* src = reinterpret_cast<const unsigned short*>(x + k0);
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            const uint32_t lo = k0 + 2 * j < K ? __ldg(src + 2 * j) : 0u, hi = k0 + 2 * j + 1 < K ? __ldg(src + 2 * j + 1) : 0u;
            w[j] = lo | (hi << 16);
        }
    }
}
// Step of a column and its inverse.  Magnitudes are compared as bit patterns (same order as the values): a NaN or an
// infinity, whose exponent field is all ones, counts as the largest and makes the step NaN, so every product with
// the column, and with it every output row that reads the column, comes out NaN instead of a finite, wrong number.
__device__ __forceinline__ float column_step(const uint32_t (&w)[12], float& inv) {
    uint32_t m = w[0] & 0x7FFF7FFFu;
#pragma unroll
    for (int j = 1; j < 12; ++j) m = __vmaxu2(m, w[j] & 0x7FFF7FFFu);
    const uint32_t top = max(m & 0xFFFFu, m >> 16);
    const uint32_t bits = __float_as_uint(__half2float(__ushort_as_half(static_cast<unsigned short>(top))));
    const bool finite = top < 0x7C00u, some = finite && top != 0u;
    const uint32_t e = bits >> 23;  // biased float exponent of the largest
    inv = some ? __uint_as_float((276u - e) << 23) : 0.f;
    return !finite ? __uint_as_float(0x7FC00000u) : (some ? __uint_as_float((e - 22u) << 23) : 0.f);
}
// rint(x inv) of the low (HIGH = false) or high half of a pair: |x| inv + 2^23 rounds to the integer |q| in the
// mantissa (|q| < 2^23), then the sign.  If the column is not finite, inv is 0 and the result arbitrary (the step is NaN).
template <bool HIGH>
__device__ __forceinline__ uint32_t quantise_value(uint32_t w, float inv) {
    const uint32_t h = HIGH ? w >> 16 : w & 0xFFFFu;
    const float a = __half2float(__ushort_as_half(static_cast<unsigned short>(h & 0x7FFFu)));
    const uint32_t q = __float_as_uint(fmaf(a, inv, 8388608.f)) - 0x4B000000u;
    const uint32_t s = uint32_t(int32_t(HIGH ? w : w << 16) >> 31);
    return (q ^ s) - s;
}
// The three plane words of four values.
__device__ __forceinline__ void split_planes(uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3, uint32_t& hi, uint32_t& mid,
                                             uint32_t& lo) {
    const uint32_t a = prmt(q0, q1, 0x5140u), b = prmt(q2, q3, 0x5140u);
    lo = prmt(a, b, 0x5410u);
    mid = prmt(a, b, 0x7632u);
    hi = prmt(prmt(q0, q1, 0x0062u), prmt(q2, q3, 0x0062u), 0x5410u);
}
// Plane words 2 s and 2 s + 1 of section s, from its four pairs, in the decoder's order.
__device__ __forceinline__ void quantise_section(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, float inv, uint32_t (&hi)[2],
                                                 uint32_t (&mid)[2], uint32_t (&lo)[2]) {
    static_assert(word_coordinate(0, 0) == 2 && word_coordinate(0, 1) == 6 && word_coordinate(0, 2) == 3 && word_coordinate(0, 3) == 7 &&
                      word_coordinate(1, 0) == 0 && word_coordinate(1, 1) == 4 && word_coordinate(1, 2) == 1 && word_coordinate(1, 3) == 5,
                  "pairs 1 and 3, then 0 and 2");
    split_planes(quantise_value<false>(w1, inv), quantise_value<false>(w3, inv), quantise_value<true>(w1, inv),
                 quantise_value<true>(w3, inv), hi[0], mid[0], lo[0]);
    split_planes(quantise_value<false>(w0, inv), quantise_value<false>(w2, inv), quantise_value<true>(w0, inv),
                 quantise_value<true>(w2, inv), hi[1], mid[1], lo[1]);
}
__device__ __forceinline__ void quantise_column(const __half* __restrict__ x, int K, int c, uint32_t out[20]) {
    uint32_t w[12];
    load_column(x, K, c, w);
    float inv;
    const float step = column_step(w, inv);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t hi[2], mid[2], lo[2];
        quantise_section(w[4 * s], w[4 * s + 1], w[4 * s + 2], w[4 * s + 3], inv, hi, mid, lo);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            out[2 * s + k] = hi[k];
            out[6 + 2 * s + k] = mid[k];
            out[12 + 2 * s + k] = lo[k];
        }
    }
    out[18] = __float_as_uint(step);
    out[19] = 0u;
}
// The planned list's record of a column, from that: the upper two planes as sixteen bits, two values to a word (words 2 k
// and 2 k + 1: the four values of word k), then the low plane, step and spare word as they were.
__device__ __forceinline__ void pair_planes(uint32_t (&q)[20]) {
    uint32_t hi[12];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        hi[2 * k] = prmt(q[k], q[6 + k], 0x1504u);
        hi[2 * k + 1] = prmt(q[k], q[6 + k], 0x3726u);
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) q[k] = hi[k];
}

}  // namespace tetra
