// Encoder search (Sec. 3.1, Eq. (2)): for a block of 24 weights, the point of the format's codebook whose
// direction is closest to the block, and the gain bit.
//
// The paper's own search is not exhaustive and runs on a CPU; this kernel computes the exact optimum of the
// same objective,  max <w, y> / (|w| |y|)  over all 2^47 indices, without visiting the rows of the lists one by
// one.  Facts of the format that it uses:
//   * Rank rows.  With weights 0, 1, 3, 6, 10 for ranks 0..4 a row's cost is 8 + 8 W, W the sum of its eight
//     ranks' weights, and its class is the parity of W.  A list is therefore every row of class cls up to some
//     W plus, of the next shell, the rows up to a limit in the order of the packed row value (the tie rule of
//     the sort):  sections 0 and 2 hold W <= 8 and W = 10 up to 0x11030011 (class 0), W <= 9 and W = 11 up to
//     0x00222011 (class 1); the middle list holds W <= 6 and W = 8 up to 0x30001010 (class 0), W <= 7 (class 1).
//     tetra_build_table checks these limits.
//   * Halves.  Rank vectors of coordinates 0..3 and 4..7 combine freely except for those limits, so the best
//     correlation of a section for (pattern byte, class, squared norm) is a maximum of sums of two half-table
//     entries (best correlation of a half for its pattern nibble, weight, norm); "row <= limit" is "high half
//     below the limit's" (a table of its own) or "equal, and low half up to the limit's" (a few entries).
//   * Norms.  A section's squared norm is 16 k + r, r in {0, 8} fixed by (parity, byte, class).  At odd parity
//     it is the row's cost, so W gives it; at even parity a coordinate adds kappa(pattern bit, rank) =
//     0,1,1,4,4 or 0,0,2,2,6 to k, and the byte floor(ones / 4).
//   * Trellis.  An even-weight byte up to complement is h(alpha) + h'(xi), alpha and xi of three bits each; the
//     codewords are exactly the triples (alpha, xi), (beta, xi), (alpha + beta, xi) with any complements.  So the
//     sections' tables hold 64 rows, and joining sections 1 and 2 is, for every xi, an XOR convolution over eight
//     alphas.  At even parity r = 8 exactly where |h(alpha) & h'(xi)| is odd, a bilinear form.
// 192 threads work on one block of weights: half tables (a thread per section, half and nibble; both parities), section
// tables (a thread per section and byte pair), join and objective (a thread per end state and class parity: four warps
// the even parity, two the odd one), then the winner is traced back through the same tables, a warp per section and
// byte of its pair.  Every sum is formed in the same order wherever it is needed, so the trace matches floats exactly.
//
// All of it is straight-line code on registers, some 8,000 instructions a block, and what it ran into was the
// instruction fetch, not the arithmetic: a CTA therefore takes three blocks in step (one SM), and code that differs
// between sections only by a constant exists once.  24,576 Gaussian blocks: 61.2 ms by scanning the rows of the
// lists in shared memory; 4.9 ms with these tables and one block per CTA; 2.3 ms three blocks in step; 1.86 ms with
// two candidates per maximum and the trace once per block; 1.65 ms with the odd parity beside the even one; 1.55 ms
// with packed additions; 1.45 ms with one copy of the half-table code; 1.30 ms with five barriers a turn instead of eight, the
// winner's warp tracing it and everything a turn ahead that can be (35,500 warp-instructions a block, issue slots
// 58 % busy; what is left is instruction fetch and the barriers between the phases).
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "../../include/tetra.h"
#include "tetra_device.cuh"
#include "tetra_launch.h"
#include "tetra_tables.h"

namespace tetra {
namespace {

constexpr int kEncThreads = 192;   // per block of weights
constexpr int kEncGroups = 3;      // blocks of weights a CTA works on, in step
constexpr float kNeg = -1.0e30f;

// ---------------------------------------------------------------------------
// compile-time shapes of the tables
// ---------------------------------------------------------------------------
constexpr int kMaxW = 11;   // largest weight of a half
constexpr int kMaxK = 9;    // largest k of a section (even parity)

__host__ __device__ constexpr int rank_weight(int r) { return r * (r + 1) / 2; }
__host__ __device__ constexpr int kappa(int c, int r) {
    const int t = (r + 1) / 2;                       // y = +-4 t (c = 0) or 2 -+ 4 t (c = 1)
    return c == 0 ? t * t : ((r & 1) ? t * t - t : t * t + t);
}

// Which (weight, kappa) cells can occur after j coordinates of a half, whatever the pattern bits.
struct Cells {
    bool v[5][kMaxW + 1][kMaxK + 1];
};
constexpr Cells free_cells() {
    Cells C{};
    C.v[0][0][0] = true;
    for (int j = 0; j < 4; ++j)
        for (int w = 0; w <= kMaxW; ++w)
            for (int k = 0; k <= kMaxK; ++k)
                if (C.v[j][w][k])
                    for (int r = 0; r < 5; ++r)
                        for (int c = 0; c < 2; ++c) {
                            const int w2 = w + rank_weight(r), k2 = k + kappa(c, r);
                            if (w2 <= kMaxW && k2 <= kMaxK) C.v[j + 1][w2][k2] = true;
                        }
    return C;
}
constexpr Cells kFree = free_cells();
// The same for vectors whose packed value is below (or, with `equal`, up to) that of the digits d0 (lowest) .. d3.
constexpr Cells prefix_cells(int d0, int d1, int d2, int d3, bool equal) {
    Cells C{};
    const int d[4] = {d0, d1, d2, d3};
    C.v[0][0][0] = equal;
    for (int j = 0; j < 4; ++j)
        for (int w = 0; w <= kMaxW; ++w)
            for (int k = 0; k <= kMaxK; ++k)
                for (int r = 0; r <= d[j]; ++r)
                    for (int c = 0; c < 2; ++c) {
                        const bool from = r < d[j] ? kFree.v[j][w][k] : C.v[j][w][k];
                        const int w2 = w + rank_weight(r), k2 = k + kappa(c, r);
                        if (from && w2 <= kMaxW && k2 <= kMaxK) C.v[j + 1][w2][k2] = true;
                    }
    return C;
}
// The limits of the partial shells, as (high half digits, low half digits), lowest coordinate first.
struct Limit {
    int hi[4], lo[4];
};
constexpr Limit kLimit0{{3, 0, 1, 1}, {1, 1, 0, 0}};    // class 0, sections 0 and 2: 0x11030011, W = 10
constexpr Limit kLimit1{{2, 2, 0, 0}, {1, 1, 0, 2}};    // class 1, sections 0 and 2: 0x00222011, W = 11
constexpr Limit kLimitM{{0, 0, 0, 3}, {0, 1, 0, 1}};    // class 0, middle section:   0x30001010, W = 8
constexpr int half_value(const int (&d)[4]) { return d[0] | (d[1] << 4) | (d[2] << 8) | (d[3] << 12); }
constexpr int half_weight(const int (&d)[4]) {
    return rank_weight(d[0]) + rank_weight(d[1]) + rank_weight(d[2]) + rank_weight(d[3]);
}
static_assert(((uint32_t(half_value(kLimit0.hi)) << 16) | uint32_t(half_value(kLimit0.lo))) == kLastRowClass0, "limit");
static_assert(((uint32_t(half_value(kLimit1.hi)) << 16) | uint32_t(half_value(kLimit1.lo))) == kLastRowClass1, "limit");
static_assert(((uint32_t(half_value(kLimitM.hi)) << 16) | uint32_t(half_value(kLimitM.lo))) == kLastRowMiddle0, "limit");
static_assert(half_weight(kLimit0.hi) == 8 && half_weight(kLimit0.lo) == 2, "limit shell");
static_assert(half_weight(kLimit1.hi) == 6 && half_weight(kLimit1.lo) == 5, "limit shell");
static_assert(half_weight(kLimitM.hi) == 6 && half_weight(kLimitM.lo) == 2, "limit shell");
constexpr Cells cells_of(const int (&d)[4], bool equal) { return prefix_cells(d[0], d[1], d[2], d[3], equal); }
constexpr Cells kLess0 = cells_of(kLimit0.hi, false), kLess1 = cells_of(kLimit1.hi, false), kLessM = cells_of(kLimitM.hi, false);
constexpr Cells kUpTo0 = cells_of(kLimit0.lo, true), kUpTo1 = cells_of(kLimit1.lo, true), kUpToM = cells_of(kLimitM.lo, true);

// Tables of a nibble at even parity.  High half: one entry per possible cell, weights 0..9 without restriction
// (H), 0..10 below limit 0 or limit M (A), 0..11 below limit 1 (B), then the limits' own correlations.  Low
// half: for every W the best over weights W, W - 2, ... (C: only the parity of the weight and an upper bound
// matter), then the entries of the limits' low halves.
constexpr int cells_before(const Cells& C, int max_w, int w, int k) {
    int n = 0;
    for (int a = 0; a <= max_w; ++a)
        for (int b = 0; b <= kMaxK; ++b) {
            if (a == w && b == k) return n;
            if (C.v[4][a][b]) ++n;
        }
    return n;
}
constexpr int cells_total(const Cells& C, int max_w) { return cells_before(C, max_w, kMaxW + 1, 0); }
constexpr int c_last(int W) {  // largest kappa over the weights W, W - 2, ...
    int m = 0;
    for (int a = W; a >= 0; a -= 2)
        for (int b = 0; b <= kMaxK; ++b)
            if (kFree.v[4][a][b] && b > m) m = b;
    return m;
}
constexpr int c_offset(int W) {
    int n = 0;
    for (int a = 0; a < W; ++a) n += c_last(a) + 1;
    return n;
}
constexpr Cells kLess0orM = [] {
    Cells C = kLess0;
    for (int w = 0; w <= kMaxW; ++w)
        for (int k = 0; k <= kMaxK; ++k) C.v[4][w][k] = C.v[4][w][k] || (kLessM.v[4][w][k] && w <= 8);
    return C;
}();
constexpr int kOffA = cells_total(kFree, 9), kOffB = kOffA + cells_total(kLess0orM, 10);
constexpr int kOffHs = kOffB + cells_total(kLess1, 11);   // correlations of the limits' high halves: 0 (or M), 1
constexpr int kHiStride = (kOffHs + 2) | 1;               // odd: a warp's nibbles fall into different banks
constexpr int kOffRes0 = c_offset(kMaxW + 1);             // low halves up to limit 0 (or M), by kappa 0..2
constexpr int kOffRes1 = kOffRes0 + 3;                    // low halves up to limit 1, by kappa 0..4
constexpr int kLoStride = (kOffRes1 + 5) | 1;
template <int W, int K> constexpr int kAtH = cells_before(kFree, 9, W, K);
template <int W, int K> constexpr int kAtA = kOffA + cells_before(kLess0orM, 10, W, K);
template <int W, int K> constexpr int kAtB = kOffB + cells_before(kLess1, 11, W, K);
template <int W> constexpr int kAtC = c_offset(W);
template <int W> constexpr int kLastC = c_last(W);
constexpr int kCells = c_offset(kMaxW + 1);

// Tables of a nibble at odd parity (the weight is the norm): low L[0..11], limits 0 or M, 1; high H[0..9],
// A[0..10], B[0..11], limits.
constexpr int kOddLoStride = 15;                          // 12 + 2, odd
constexpr int kOddOffA = 10, kOddOffB = 21, kOddOffHs = 33, kOddHiStride = 35;

// Half vectors for the trace, weight <= 11: value | weight << 16.
struct HalfList {
    uint32_t v[176];
    int n;
};
constexpr HalfList half_list() {
    HalfList L{};
    for (int code = 0; code < 625; ++code) {
        const int d[4] = {code % 5, (code / 5) % 5, (code / 25) % 5, code / 125};
        const int w = half_weight(d);
        if (w <= kMaxW) L.v[L.n++] = uint32_t(half_value(d)) | (uint32_t(w) << 16);
    }
    return L;
}
constexpr HalfList kHalfListHost = half_list();
constexpr int kHalfVectors = kHalfListHost.n;
__device__ const HalfList kHalfList = half_list();

// Where the low tables keep the best over weights W, W - 2, ...: offset | largest kappa << 16.
struct LowIndex {
    uint32_t v[kMaxW + 1];
};
constexpr LowIndex low_index() {
    LowIndex L{};
    for (int w = 0; w <= kMaxW; ++w) L.v[w] = uint32_t(c_offset(w)) | (uint32_t(c_last(w)) << 16);
    return L;
}
__device__ const LowIndex kLowIndex = low_index();

template <int I, int N, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}
template <int I, typename F>
__device__ __forceinline__ void static_down(F&& f) {
    if constexpr (I >= 0) {
        f(std::integral_constant<int, I>{});
        static_down<I - 1>(f);
    }
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// (a0 + b, a1 + b) in one instruction, rounded and flushed like __fadd_rn in this file's build.
__device__ __forceinline__ void add2(float a0, float a1, float b, float& s0, float& s1) {
    uint64_t aa, bb, ss;
    asm("mov.b64 %0, {%1, %2};" : "=l"(aa) : "f"(a0), "f"(a1));
    asm("mov.b64 %0, {%1, %1};" : "=l"(bb) : "f"(b));
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(ss) : "l"(aa), "l"(bb));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(s0), "=f"(s1) : "l"(ss));
}

// ---------------------------------------------------------------------------
// shared memory of a CTA
// ---------------------------------------------------------------------------
constexpr int kRow = 12;     // floats per section-table row at even parity (k, or k + 1, from 0; the rest absent)
constexpr int kOddRow = 8;   // at odd parity: index W / 2, 0..5
struct EncShared {
    float lo[3][16 * kLoStride];
    float hi[3][16 * kHiStride];
    float lo_odd[3][16 * kOddLoStride];
    float hi_odd[3][16 * kOddHiStride];
    // section tables, even and odd parity: [section][class][pair = alpha + 8 xi][row]
    alignas(16) float F[3][2][64 * kRow];
    alignas(16) float O[3][2][64 * kOddRow];
    float rs[32];             // 1 / sqrt(16 m)
    float w[2][24];           // this turn's and the next one's
    uint32_t halves[kHalfVectors];
    uint32_t low_index[kMaxW + 1];
    uint8_t bytes[64];        // h(alpha) + h'(xi)
    float red_val[6];         // per warp: the best of the objective
    uint32_t red_arg[6];      // and the thread that holds it
    float win_H[20];
    float win_G;
    int win_arg, win_par;
    // the winner so far, per section: byte pair, class, index and value of its table entry
    int hit_pair[3], hit_cls[3], hit_k[3];
    float hit_target[3];
    float out_val, out_wn2;   // of the traced block: the best of the objective, the squared norm of its weights
    int out_live, out_even;
    // its row, looked for with the pair's byte and with its complement: index inside the section's list, or none
    uint32_t found_row[3][2];
    bool found[3][2];
};
static_assert(sizeof(EncShared) * kEncGroups <= 226 * 1024, "one CTA per SM");

// h(a), a < 8, and h'(x), x < 8: representatives of the bytes of the two [8,4] codes up to complement.
__device__ __forceinline__ uint32_t hamming_byte(uint32_t v, uint32_t b0, uint32_t b1, uint32_t b2) {
    return ((v & 1) ? b0 : 0u) ^ ((v & 2) ? b1 : 0u) ^ ((v & 4) ? b2 : 0u);
}
__device__ __forceinline__ uint32_t pair_byte(int pair) {
    return hamming_byte(uint32_t(pair) & 7u, 0x8Bu, 0x96u, 0xACu) ^ hamming_byte(uint32_t(pair) >> 3, 0x8Du, 0x9Au, 0xB4u);
}
// 1 where the squared norm of a section with this byte is 8 modulo 16 at even parity (byte and complement alike)
__device__ __forceinline__ int odd_overlap(uint32_t byte) { return (__popc(byte) >> 1) & 1; }

// At even parity a coordinate with a pattern bit adds 4 to the squared norm besides 16 kappa: k = kappa + this.
__device__ __forceinline__ int ones_offset(uint32_t byte) { return __popc(byte) >> 2; }

// ---------------------------------------------------------------------------
// half tables
// ---------------------------------------------------------------------------
// The five products of a coordinate, w y(rank): the trace forms them the same way.
__device__ __forceinline__ void products_even(float w, int c, float (&a)[5]) {
    a[0] = __fmul_rn(w, c ? 2.f : 0.f);
    a[1] = __fmul_rn(w, c ? -2.f : 4.f);
    a[2] = __fmul_rn(w, c ? 6.f : -4.f);
    a[3] = __fmul_rn(w, c ? -6.f : 8.f);
    a[4] = __fmul_rn(w, c ? 10.f : -8.f);
}
__device__ __forceinline__ void products_odd(float w, int c, float (&a)[5]) {
    const float s = c ? -w : w;
    a[0] = s;
    a[1] = __fmul_rn(s, -3.f);
    a[2] = __fmul_rn(s, 5.f);
    a[3] = __fmul_rn(s, -7.f);
    a[4] = __fmul_rn(s, 9.f);
}

// One step of the prefix-limited table (before the free table takes the same step): vectors below the digits so
// far = a smaller digit after anything, or the same digit after a smaller prefix.
template <int J, int D, const Cells& PC>
__device__ __forceinline__ void prefix_step(const float (&F)[kMaxW + 1][kMaxK + 1], float (&P)[kMaxW + 1][kMaxK + 1],
                                            const float (&a)[5], int c) {
    static_down<kMaxW>([&](auto wi) {
        constexpr int W = decltype(wi)::value;
        static_down<kMaxK>([&](auto ki) {
            constexpr int K = decltype(ki)::value;
            if constexpr (PC.v[J + 1][W][K]) {
                float v = kNeg;
                static_for<0, D + 1>([&](auto ri) {
                    constexpr int R = decltype(ri)::value;
                    if constexpr (W >= rank_weight(R)) {
                        constexpr int W0 = W - rank_weight(R), K0 = K - kappa(0, R), K1 = K - kappa(1, R);
                        constexpr bool f0 = K0 >= 0 && (R < D ? kFree.v[J][W0][K0 < 0 ? 0 : K0] : PC.v[J][W0][K0 < 0 ? 0 : K0]);
                        constexpr bool f1 = K1 >= 0 && (R < D ? kFree.v[J][W0][K1 < 0 ? 0 : K1] : PC.v[J][W0][K1 < 0 ? 0 : K1]);
                        if constexpr (f0 || f1) {
                            float s0 = kNeg, s1 = kNeg;
                            if constexpr (f0) s0 = R < D ? F[W0][K0] : P[W0][K0];
                            if constexpr (f1) s1 = R < D ? F[W0][K1] : P[W0][K1];
                            v = fmaxf(v, __fadd_rn(K0 == K1 ? s0 : (c ? s1 : s0), a[R]));
                        }
                    }
                });
                P[W][K] = v;
            }
        });
    });
}
template <int J>
__device__ __forceinline__ void free_step(float (&F)[kMaxW + 1][kMaxK + 1], const float (&a)[5], int c) {
    static_down<kMaxW>([&](auto wi) {
        constexpr int W = decltype(wi)::value;
        static_down<kMaxK>([&](auto ki) {
            constexpr int K = decltype(ki)::value;
            if constexpr (kFree.v[J + 1][W][K]) {
                float v = kNeg;
                static_for<0, 5>([&](auto ri) {
                    constexpr int R = decltype(ri)::value;
                    if constexpr (W >= rank_weight(R)) {
                        constexpr int W0 = W - rank_weight(R), K0 = K - kappa(0, R), K1 = K - kappa(1, R);
                        constexpr bool f0 = K0 >= 0 && kFree.v[J][W0][K0 < 0 ? 0 : K0];
                        constexpr bool f1 = K1 >= 0 && kFree.v[J][W0][K1 < 0 ? 0 : K1];
                        if constexpr (f0 || f1) {
                            float s0 = kNeg, s1 = kNeg;
                            if constexpr (f0) s0 = F[W0][K0];
                            if constexpr (f1) s1 = F[W0][K1];
                            v = fmaxf(v, __fadd_rn(K0 == K1 ? s0 : (c ? s1 : s0), a[R]));
                        }
                    }
                });
                F[W][K] = v;
            }
        });
    });
}

// Even parity: the tables of (section, half, nibble).  w4: the half's four weights; mid: the middle section, whose list
// has its own limit (M instead of 0 and 1; what the other limits give is not read there).  One copy of this code for
// all sections: straight-line code is fetched more slowly than it runs.
template <bool HIGH>
__device__ __forceinline__ void half_even(const float* w4, int nibble, bool mid, float* out) {
    float F[kMaxW + 1][kMaxK + 1], A[kMaxW + 1][kMaxK + 1], B[kMaxW + 1][kMaxK + 1], M[kMaxW + 1][kMaxK + 1];
    F[0][0] = 0.f;
    A[0][0] = 0.f;   // only the "up to" tables read it
    B[0][0] = 0.f;
    M[0][0] = 0.f;
    float hs0 = 0.f, hs1 = 0.f, hsm = 0.f;  // correlations of the limits' high halves
    static_for<0, 4>([&](auto ji) {
        constexpr int J = decltype(ji)::value;
        const int c = (nibble >> J) & 1;
        float a[5];
        products_even(w4[J], c, a);
        if constexpr (HIGH) {
            constexpr int D0 = kLimit0.hi[J], D1 = kLimit1.hi[J], DM = kLimitM.hi[J];  // digits of the limits' high halves
            prefix_step<J, kLimit0.hi[J], kLess0>(F, A, a, c);
            prefix_step<J, kLimit1.hi[J], kLess1>(F, B, a, c);
            prefix_step<J, kLimitM.hi[J], kLessM>(F, M, a, c);
            hs0 = __fadd_rn(hs0, a[D0]);
            hs1 = __fadd_rn(hs1, a[D1]);
            hsm = __fadd_rn(hsm, a[DM]);
        } else {
            prefix_step<J, kLimit0.lo[J], kUpTo0>(F, A, a, c);
            prefix_step<J, kLimit1.lo[J], kUpTo1>(F, B, a, c);
            prefix_step<J, kLimitM.lo[J], kUpToM>(F, M, a, c);
        }
        free_step<J>(F, a, c);
    });
    if constexpr (HIGH) {
        static_for<0, kMaxW + 1>([&](auto wi) {
            constexpr int W = decltype(wi)::value;
            static_for<0, kMaxK + 1>([&](auto ki) {
                constexpr int K = decltype(ki)::value;
                if constexpr (W <= 9 && kFree.v[4][W][K]) out[kAtH<W, K>] = F[W][K];
                if constexpr (W <= 10 && kLess0orM.v[4][W][K]) {
                    float v0 = kNeg, vm = kNeg;
                    if constexpr (kLess0.v[4][W][K]) v0 = A[W][K];
                    if constexpr (kLessM.v[4][W][K]) vm = M[W][K];
                    out[kAtA<W, K>] = mid ? vm : v0;
                }
                if constexpr (kLess1.v[4][W][K]) out[kAtB<W, K>] = B[W][K];
            });
        });
        out[kOffHs] = mid ? hsm : hs0;
        out[kOffHs + 1] = hs1;
    } else {
        static_for<0, 2>([&](auto pi) {
            float best[kMaxK + 1];
#pragma unroll
            for (int k = 0; k <= kMaxK; ++k) best[k] = kNeg;
            static_for<0, (kMaxW + 1) / 2>([&](auto ii) {
                constexpr int W = 2 * decltype(ii)::value + decltype(pi)::value;
                static_for<0, kLastC<W> + 1>([&](auto ki) {
                    constexpr int K = decltype(ki)::value;
                    if constexpr (kFree.v[4][W][K]) best[K] = fmaxf(best[K], F[W][K]);
                    out[kAtC<W> + K] = best[K];
                });
            });
        });
        static_for<0, 5>([&](auto ki) {
            constexpr int K = decltype(ki)::value;
            if constexpr (K < 3) {
                float v0 = kNeg, vm = kNeg;
                if constexpr (kUpTo0.v[4][2][K]) v0 = A[2][K];
                if constexpr (kUpToM.v[4][2][K]) vm = M[2][K];
                out[kOffRes0 + K] = mid ? vm : v0;
            }
            float v1 = kNeg;
            if constexpr (kUpTo1.v[4][5][K]) v1 = B[5][K];
            out[kOffRes1 + K] = v1;
        });
    }
}

// Odd parity: the same with the weight as the only index.
constexpr bool odd_cell_at(const Cells& C, int j, int w) {
    for (int k = 0; k <= kMaxK; ++k)
        if (C.v[j][w][k]) return true;
    return false;
}
template <const Cells& C, int J, int W> constexpr bool kOddCell = odd_cell_at(C, J, W);
template <int J, int D, const Cells& PC>
__device__ __forceinline__ void odd_prefix_step(const float (&F)[kMaxW + 1], float (&P)[kMaxW + 1], const float (&a)[5]) {
    static_down<kMaxW>([&](auto wi) {
        constexpr int W = decltype(wi)::value;
        if constexpr (kOddCell<PC, J + 1, W>) {
            float v = kNeg;
            static_for<0, D + 1>([&](auto ri) {
                constexpr int R = decltype(ri)::value;
                if constexpr (W >= rank_weight(R)) {
                    constexpr int W0 = W - rank_weight(R);
                    if constexpr (R < D) {
                        if constexpr (kOddCell<kFree, J, W0>) v = fmaxf(v, __fadd_rn(F[W0], a[R]));
                    } else {
                        if constexpr (kOddCell<PC, J, W0>) v = fmaxf(v, __fadd_rn(P[W0], a[R]));
                    }
                }
            });
            P[W] = v;
        }
    });
}
template <bool HIGH, bool MID>
__device__ __forceinline__ void half_odd(const float* w4, int nibble, float* out) {
    float F[kMaxW + 1], A[kMaxW + 1], B[kMaxW + 1];
#pragma unroll
    for (int w = 0; w <= kMaxW; ++w) F[w] = A[w] = B[w] = kNeg;
    F[0] = A[0] = B[0] = 0.f;
    float hs0 = 0.f, hs1 = 0.f;
    static_for<0, 4>([&](auto ji) {
        constexpr int J = decltype(ji)::value;
        [[maybe_unused]] constexpr int D0 = kLimit0.hi[J], D1 = kLimit1.hi[J], DM = kLimitM.hi[J];  // digits of the limits' high halves
        float a[5];
        products_odd(w4[J], (nibble >> J) & 1, a);
        if constexpr (HIGH) {
            if constexpr (MID) {
                odd_prefix_step<J, kLimitM.hi[J], kLessM>(F, A, a);
                hs0 = __fadd_rn(hs0, a[DM]);
            } else {
                odd_prefix_step<J, kLimit0.hi[J], kLess0>(F, A, a);
                odd_prefix_step<J, kLimit1.hi[J], kLess1>(F, B, a);
                hs0 = __fadd_rn(hs0, a[D0]);
                hs1 = __fadd_rn(hs1, a[D1]);
            }
        } else {
            if constexpr (MID) {
                odd_prefix_step<J, kLimitM.lo[J], kUpToM>(F, A, a);
            } else {
                odd_prefix_step<J, kLimit0.lo[J], kUpTo0>(F, A, a);
                odd_prefix_step<J, kLimit1.lo[J], kUpTo1>(F, B, a);
            }
        }
        static_down<kMaxW>([&](auto wi) {
            constexpr int W = decltype(wi)::value;
            if constexpr (kOddCell<kFree, J + 1, W>) {
                float v = kNeg;
                static_for<0, 5>([&](auto ri) {
                    constexpr int R = decltype(ri)::value;
                    if constexpr (W >= rank_weight(R)) {
                        constexpr int W0 = W - rank_weight(R);
                        if constexpr (kOddCell<kFree, J, W0>) v = fmaxf(v, __fadd_rn(F[W0], a[R]));
                    }
                });
                F[W] = v;
            }
        });
    });
    if constexpr (HIGH) {
        static_for<0, kMaxW + 1>([&](auto wi) {
            constexpr int W = decltype(wi)::value;
            if constexpr (W <= 9) out[W] = F[W];
            if constexpr (W <= 10) {
                float v = kNeg;
                if constexpr (MID ? kOddCell<kLessM, 4, W> : kOddCell<kLess0, 4, W>) v = A[W];
                out[kOddOffA + W] = v;
            }
            float v = kNeg;
            if constexpr (!MID && kOddCell<kLess1, 4, W>) v = B[W];
            out[kOddOffB + W] = v;
        });
        out[kOddOffHs] = hs0;
        out[kOddOffHs + 1] = hs1;
    } else {
#pragma unroll
        for (int w = 0; w <= kMaxW; ++w) out[w] = F[w];
        out[12] = A[2];
        if constexpr (!MID) out[13] = B[5];
    }
}

// ---------------------------------------------------------------------------
// section tables
// ---------------------------------------------------------------------------
// The possible kappas of a weight in a high-half table.
constexpr int cell_count(const Cells& C, int w) {
    int n = 0;
    for (int k = 0; k <= kMaxK; ++k) n += C.v[4][w][k] ? 1 : 0;
    return n;
}
constexpr int cell_nth(const Cells& C, int w, int i) {
    for (int k = 0; k <= kMaxK; ++k)
        if (C.v[4][w][k] && i-- == 0) return k;
    return -1;
}
template <const Cells& C, int W> constexpr int kCellCount = cell_count(C, W);
template <const Cells& C, int W, int I> constexpr int kCellNth = cell_nth(C, W, I);
template <int TABLE, int W, int K> constexpr int kAtHigh = TABLE == 0 ? kAtH<W, K> : (TABLE == 1 ? kAtA<W, K> : kAtB<W, K>);

// T[n] = max(T[n], h[W][k] + C[V][n - k]) over the cells k of weight W of a high-half table (TABLE 0: H, 1: A, 2: B;
// CELLS: its possible cells); two cells at a time, so that most maxima take two candidates.
template <int TABLE, const Cells& CELLS, int W, int V, int KMAX>
__device__ __forceinline__ void combine_even(const float* hi, const float (&C)[kCells], float (&T)[kMaxK + 1]) {
    constexpr int LAST = kLastC<V>;
    static_for<0, (kCellCount<CELLS, W> + 1) / 2>([&](auto ti) {
        constexpr int I = 2 * decltype(ti)::value;
        constexpr int KA = kCellNth<CELLS, W, I>, KB = kCellNth<CELLS, W, I + 1>;  // KB = -1: no second cell
        float sa[LAST + 2], sb[LAST + 2] = {};
        auto sums = [&](float h, float (&s)[LAST + 2]) {
#pragma unroll
            for (int i = 0; i < LAST; i += 2) add2(C[kAtC<V> + i], C[kAtC<V> + i + 1], h, s[i], s[i + 1]);
            if constexpr (LAST % 2 == 0) s[LAST] = __fadd_rn(h, C[kAtC<V> + LAST]);
        };
        sums(hi[kAtHigh<TABLE, W, KA>], sa);
        if constexpr (KB >= 0) sums(hi[kAtHigh<TABLE, W, KB>], sb);
        static_for<0, KMAX + 1>([&](auto ni) {
            constexpr int N = decltype(ni)::value;
            constexpr bool a = N >= KA && N - KA <= LAST, b = KB >= 0 && N >= KB && N - KB <= LAST;
            if constexpr (a && b) T[N] = max3(T[N], sa[N - KA], sb[N - KB]);
            else if constexpr (a) T[N] = fmaxf(T[N], sa[N - KA]);
            else if constexpr (b) T[N] = fmaxf(T[N], sb[N - KB]);
        });
    });
}

template <bool MID>
__device__ __forceinline__ void section_even(const float* lo, const float* hi, float (&T0)[kMaxK + 1], float (&T1)[kMaxK + 1]) {
    float C[kCells];
#pragma unroll
    for (int i = 0; i < kCells; ++i) C[i] = lo[i];
    static_for<0, kMaxW + 1>([&](auto wi) {
        constexpr int W = decltype(wi)::value;
        if constexpr (MID) {
            if constexpr (W <= 7) combine_even<0, kFree, W, 7 - W, 7>(hi, C, T1);
            if constexpr (W <= 8) combine_even<1, kLessM, W, 8 - W, kMaxK - 1>(hi, C, T0);
        } else {
            if constexpr (W <= 9) combine_even<0, kFree, W, 9 - W, kMaxK>(hi, C, T1);
            if constexpr (W <= 8) combine_even<0, kFree, W, 8 - W, kMaxK - 1>(hi, C, T0);
            if constexpr (W <= 10) combine_even<1, kLess0, W, 10 - W, kMaxK - 1>(hi, C, T0);
            combine_even<2, kLess1, W, 11 - W, kMaxK>(hi, C, T1);
        }
    });
}

// kappa of the limits' high halves for a pattern nibble
__device__ __forceinline__ int kappa_hs(int which, int nibble) {  // which: 0, 1 or 2 = M
    const int c0 = nibble & 1, c1 = (nibble >> 1) & 1, c2 = (nibble >> 2) & 1, c3 = (nibble >> 3) & 1;
    if (which == 0) return (c0 ? 2 : 4) + (c2 ? 0 : 1) + (c3 ? 0 : 1);
    if (which == 1) return (c0 ? 2 : 1) + (c1 ? 2 : 1);
    return c3 ? 2 : 4;
}

template <bool MID>
__device__ __forceinline__ void section_odd(const float* lo, const float* hi, float (&T)[kMaxW + 1]) {
    float L[kMaxW + 1];
#pragma unroll
    for (int w = 0; w <= kMaxW; ++w) L[w] = lo[w];
    constexpr int FULL = MID ? 7 : 9;
#pragma unroll
    for (int wh = 0; wh <= FULL; ++wh) {
        const float h = hi[wh];
#pragma unroll
        for (int wl = 0; wl <= FULL - wh; ++wl) T[wh + wl] = fmaxf(T[wh + wl], __fadd_rn(h, L[wl]));
    }
    if constexpr (MID) {
#pragma unroll
        for (int wh = 0; wh <= 8; ++wh) T[8] = fmaxf(T[8], __fadd_rn(hi[kOddOffA + wh], L[8 - wh]));
        T[8] = fmaxf(T[8], __fadd_rn(hi[kOddOffHs], lo[12]));
    } else {
#pragma unroll
        for (int wh = 0; wh <= 10; ++wh) T[10] = fmaxf(T[10], __fadd_rn(hi[kOddOffA + wh], L[10 - wh]));
        T[10] = fmaxf(T[10], __fadd_rn(hi[kOddOffHs], lo[12]));
        static_for<0, kMaxW + 1>([&](auto wi) {
            constexpr int WH = decltype(wi)::value;
            if constexpr (kOddCell<kLess1, 4, WH>) T[11] = fmaxf(T[11], __fadd_rn(hi[kOddOffB + WH], L[11 - WH]));
        });
        T[11] = fmaxf(T[11], __fadd_rn(hi[kOddOffHs + 1], lo[13]));
    }
}

// The section tables of one section, thread = byte pair.  EVEN: rows of k; else rows of W / 2.
template <bool EVEN, bool MID>
__device__ __forceinline__ void section_rows(EncShared& S, int s, int pair) {
    float* rows0 = EVEN ? S.F[s][0] : S.O[s][0];
    float* rows1 = EVEN ? S.F[s][1] : S.O[s][1];
    const uint32_t byte = S.bytes[pair];
    if constexpr (EVEN) {
        float* r0 = rows0 + pair * kRow;
        float* r1 = rows1 + pair * kRow;
#pragma unroll
        for (int k = 0; k < kRow; ++k) r0[k] = r1[k] = kNeg;
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            const uint32_t b = e ? byte ^ 0xFFu : byte;
            float T0[kMaxK + 1], T1[kMaxK + 1];
#pragma unroll
            for (int k = 0; k <= kMaxK; ++k) T0[k] = T1[k] = kNeg;
            section_even<MID>(S.lo[s] + (b & 15u) * kLoStride, S.hi[s] + (b >> 4) * kHiStride, T0, T1);
            const int up = ones_offset(b);
#pragma unroll
            for (int k = 0; k <= kMaxK; ++k) {
                if (k < kMaxK) r0[up + k] = fmaxf(r0[up + k], T0[k]);
                r1[up + k] = fmaxf(r1[up + k], T1[k]);
            }
        }
        // the rows whose high half IS a limit's: their norms depend on the nibble, so they are added in place
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            const uint32_t b = e ? byte ^ 0xFFu : byte;
            const float* lo = S.lo[s] + (b & 15u) * kLoStride;
            const float* hi = S.hi[s] + (b >> 4) * kHiStride;
            const float h0 = hi[kOffHs];
            const int k0 = kappa_hs(MID ? 2 : 0, int(b >> 4)) + ones_offset(b);
            if constexpr (MID) r0[k0] = fmaxf(r0[k0], __fadd_rn(h0, lo[kAtC<0>]));  // 0x30000000, W = 6
#pragma unroll
            for (int k = 0; k < 3; ++k) r0[k0 + k] = fmaxf(r0[k0 + k], __fadd_rn(h0, lo[kOffRes0 + k]));
            if constexpr (!MID) {
                const float h1 = hi[kOffHs + 1];
                const int k1 = kappa_hs(1, int(b >> 4)) + ones_offset(b);
#pragma unroll
                for (int k = 0; k < 5; ++k) r1[k1 + k] = fmaxf(r1[k1 + k], __fadd_rn(h1, lo[kOffRes1 + k]));
            }
        }
    } else {
        float T[kMaxW + 1];
#pragma unroll
        for (int w = 0; w <= kMaxW; ++w) T[w] = kNeg;
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
            const uint32_t b = e ? byte ^ 0xFFu : byte;
            section_odd<MID>(S.lo_odd[s] + (b & 15u) * kOddLoStride, S.hi_odd[s] + (b >> 4) * kOddHiStride, T);
        }
        float* r0 = rows0 + pair * kOddRow;
        float* r1 = rows1 + pair * kOddRow;
#pragma unroll
        for (int k = 0; k < kOddRow; ++k) {
            r0[k] = k < 6 ? T[k < 6 ? 2 * k : 0] : kNeg;
            r1[k] = k < 6 ? T[k < 6 ? 2 * k + 1 : 0] : kNeg;
        }
    }
}

// ---------------------------------------------------------------------------
// join and objective: thread = (end state gamma + 8 xi, parity `par` of the classes of sections 1 and 2)
// ---------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void load_row(const float* row, float (&v)[N]) {
    static_assert(N % 4 == 0, "whole quads");
#pragma unroll
    for (int i = 0; i < N; i += 4) {
        const float4 q = *reinterpret_cast<const float4*>(row + i);
        v[i] = q.x;
        v[i + 1] = q.y;
        v[i + 2] = q.z;
        v[i + 3] = q.w;
    }
}

// H[i + j + SHIFT] = max(., a[i] + b[j]) for i < NA, j < NB: two sums per addition, two candidates per maximum.
template <int NA, int NB, int SHIFT, int LA, int LB, int LH>
__device__ __forceinline__ void max_plus(const float (&a)[LA], const float (&b)[LB], float (&H)[LH]) {
    static_for<0, (NB + 1) / 2>([&](auto ji) {
        constexpr int j = 2 * decltype(ji)::value;
        constexpr bool two = j + 1 < NB;
        float s[2][NA + 1];
#pragma unroll
        for (int i = 0; i + 1 < NA; i += 2) {
            add2(a[i], a[i + 1], b[j], s[0][i], s[0][i + 1]);
            if constexpr (two) add2(a[i], a[i + 1], b[j + 1], s[1][i], s[1][i + 1]);
        }
        if constexpr (NA & 1) {
            s[0][NA - 1] = __fadd_rn(a[NA - 1], b[j]);
            if constexpr (two) s[1][NA - 1] = __fadd_rn(a[NA - 1], b[j + 1]);
        }
        static_for<0, NA + 1>([&](auto ii) {
            constexpr int i = decltype(ii)::value, n = i + j + SHIFT;
            if constexpr (two && i > 0 && i < NA) H[n] = max3(H[n], s[0][i], s[1][i - 1]);
            else if constexpr (i < NA) H[n] = fmaxf(H[n], s[0][i]);
            else if constexpr (two) H[n] = fmaxf(H[n], s[1][i - 1]);
        });
    });
}

constexpr int kH = 20;  // entries after two sections: norms 16 i (+ 8), i < 20

// Row lengths in use: even parity k <= 9, the middle list k <= 8 (class 0) and k <= 7.  Odd parity: W / 2 <= 5, the
// middle list 4 and 3.
template <bool EVEN, int PAR>
__device__ __forceinline__ void join_two(const EncShared& S, int gamma, int xi, bool odd_end, float (&H)[kH]) {
#pragma unroll
    for (int i = 0; i < kH; ++i) H[i] = kNeg;
#pragma unroll 1
    for (int alpha = 0; alpha < 8; ++alpha) {
        const int i = alpha + 8 * xi, j = (alpha ^ gamma) + 8 * xi;
        static_for<0, 2>([&](auto ci) {
            constexpr int c1 = decltype(ci)::value, c2 = c1 ^ PAR;
            if constexpr (EVEN) {
                // norms 16 k1 + r1 and 16 k2 + r2: index k1 + k2, plus one when both residues are 8
                const bool raised = !odd_end && odd_overlap(S.bytes[i]);
                float r[12], a[12], b[12];
                load_row(S.F[0][c1] + i * kRow, r);
                load_row(S.F[1][c2] + j * kRow, b);
                a[0] = raised ? kNeg : r[0];
#pragma unroll
                for (int k = 1; k < 12; ++k) a[k] = raised ? r[k - 1] : r[k];
                max_plus<11, c2 ? 8 : 9, 0>(a, b, H);
            } else {
                float a[8], b[8];
                load_row(S.O[0][c1] + i * kOddRow, a);
                load_row(S.O[1][c2] + j * kOddRow, b);
                max_plus<6, c2 ? 4 : 5, c1 & c2>(a, b, H);  // W1 + W2 = 2 (index) + (classes' parity)
            }
        });
    }
}

// G[n] = best correlation of all three sections at squared norm 16 (n + m0): returns the best of G / norm.
template <bool EVEN, int CLS3>
__device__ __forceinline__ void objective(const EncShared& S, int m0, int end_pair, const float (&H)[kH], float& val, float& corr, int& arg) {
    constexpr int NA = EVEN ? 19 : 10, NB = EVEN ? 10 : 6, NG = NA + NB - 1;
    float G[NG];
#pragma unroll
    for (int n = 0; n < NG; ++n) G[n] = kNeg;
    float b[EVEN ? 12 : 8];
    load_row((EVEN ? S.F[2][CLS3] : S.O[2][CLS3]) + end_pair * (EVEN ? kRow : kOddRow), b);
    max_plus<NA, NB, 0>(H, b, G);
    val = kNeg;
    corr = kNeg;
    arg = 0;
#pragma unroll
    for (int n = 0; n < NG; ++n) {
        const float v = G[n] * S.rs[n + m0];
        if (v > val) {
            val = v;
            corr = G[n];
            arg = n;
        }
    }
}

// ---------------------------------------------------------------------------
// trace of the winner: one warp per section
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool row_in_list(int section, int cls, int w, uint32_t row) {
    if (section == 1) return cls ? w <= 7 : (w <= 6 || (w == 8 && row <= kLastRowMiddle0));
    return cls ? (w <= 9 || (w == 11 && row <= kLastRowClass1)) : (w <= 8 || (w == 10 && row <= kLastRowClass0));
}
// The products of a half with the values of every rank, a lane each: lane 5 j + r holds w_j y(pattern bit j, rank r).
__device__ __forceinline__ float half_products(bool even, const float* w4, int nibble) {
    const int lane = threadIdx.x & 31, j = min(lane / 5, 3), r = lane - 5 * (lane / 5), c = (nibble >> j) & 1, t = (r + 1) >> 1;
    const int v0 = (r & 1) ? 4 * t : -4 * t;
    return __fmul_rn(w4[j], float(even ? (c ? 2 - v0 : v0) : (c ? v0 - 1 : 1 - v0)));
}
// Correlation of a half vector from those, the sum in the tables' order; all lanes.
__device__ __forceinline__ float half_corr(float products, uint32_t value) {
    float sum = __shfl_sync(0xFFFFFFFFu, products, int(value & 7u));
#pragma unroll
    for (int j = 1; j < 4; ++j) sum = __fadd_rn(sum, __shfl_sync(0xFFFFFFFFu, products, 5 * j + int((value >> (4 * j)) & 7u)));
    return sum;
}
// kappa of a half vector at even parity: four bits per rank, by pattern bit.
__device__ __forceinline__ int half_kappa(int nibble, uint32_t value) {
    constexpr uint32_t k0 = 0x44110u, k1 = 0x62200u;
    static_assert(kappa(0, 1) == 1 && kappa(0, 2) == 1 && kappa(0, 3) == 4 && kappa(0, 4) == 4 && kappa(0, 0) == 0, "kappa");
    static_assert(kappa(1, 1) == 0 && kappa(1, 2) == 2 && kappa(1, 3) == 2 && kappa(1, 4) == 6 && kappa(1, 0) == 0, "kappa");
    uint32_t kap = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) kap += (((nibble >> j) & 1 ? k1 : k0) >> ((value >> (4 * j) & 7u) * 4u)) & 15u;
    return int(kap);
}

// Looks for the row of section s whose correlation with the pair's byte (e = 0) or its complement (e = 1) is the
// winner's at its index of the section's table.
__device__ __noinline__ void trace_section(EncShared& S, const DeviceTables* __restrict__ tab, const float* w24, bool even, int s, int e) {
    const int lane = threadIdx.x & 31;
    const int cls = S.hit_cls[s], k = S.hit_k[s];
    const float target = S.hit_target[s];
    const int w_total = 2 * k + cls;  // odd parity: the row's weight
    const float* w = w24 + 8 * s;
    uint32_t row = 0;
    const uint32_t byte = S.bytes[S.hit_pair[s]] ^ (e ? 0xFFu : 0u);
    bool found = false;
    {
        const int nlo = int(byte & 15u), nhi = int(byte >> 4);
        const int kap = k - ones_offset(byte);
        const float* lo = even ? S.lo[s] + nlo * kLoStride : S.lo_odd[s] + nlo * kOddLoStride;
        // 1. a high half with a partner in the low tables
        uint32_t high = 0;
        float high_corr = 0.f;
        int high_kap = 0;
        bool have = false;
        const float high_products = half_products(even, w + 4, nhi), low_products = half_products(even, w, nlo);
        const uint32_t lim = s == 1 ? kLastRowMiddle0 >> 16 : (cls ? kLastRowClass1 >> 16 : kLastRowClass0 >> 16);
        const bool limited = !(s == 1 && cls);            // the list has a partial shell
        const int full = s == 1 ? (cls ? 7 : 6) : (cls ? 9 : 8);
#pragma unroll 1
        for (int i0 = 0; i0 < kHalfVectors && !have; i0 += 32) {
            const bool there = i0 + lane < kHalfVectors;
            const uint32_t hv = S.halves[there ? i0 + lane : 0];
            const int wh = int(hv >> 16);
            const uint32_t v = hv & 0xFFFFu;
            const float hc = half_corr(high_products, v);
            bool hit = false;
            int hk = 0;
            if (even) {
                hk = half_kappa(nhi, v);
                const int kl = kap - hk;
                auto partner = [&](int W) {  // best low half of weights W, W - 2, ...
                    const uint32_t at = S.low_index[max(W, 0)];
                    if (W >= 0 && kl >= 0 && kl <= int(at >> 16)) hit = hit || __fadd_rn(hc, lo[int(at & 0xFFFFu) + kl]) == target;
                };
                partner(full - wh);
                if (limited && v < lim) partner(full + 2 - wh);
                if (limited && v == lim) {
                    const int n = cls ? 5 : 3, off = cls ? kOffRes1 : kOffRes0;
                    if (kl >= 0 && kl < n) hit = hit || __fadd_rn(hc, lo[off + kl]) == target;
                }
            } else {
                const int wl = w_total - wh;
                if (wl >= 0) {
                    const bool whole = w_total <= full || (limited && v < lim);
                    if (whole) hit = __fadd_rn(hc, lo[wl]) == target;
                    else if (limited && v == lim) hit = __fadd_rn(hc, lo[cls ? 13 : 12]) == target;
                }
            }
            const uint32_t any = __ballot_sync(0xFFFFFFFFu, hit && there);
            if (any) {
                const int src = __ffs(int(any)) - 1;
                high = __shfl_sync(0xFFFFFFFFu, hv, src);
                high_corr = __shfl_sync(0xFFFFFFFFu, hc, src);
                high_kap = __shfl_sync(0xFFFFFFFFu, hk, src);
                have = true;
            }
        }
        // 2. the low half: sum, norm and membership decide
#pragma unroll 1
        for (int i0 = 0; i0 < kHalfVectors && have && !found; i0 += 32) {
            const bool there = i0 + lane < kHalfVectors;
            const uint32_t lv = S.halves[there ? i0 + lane : 0];
            const float lc = half_corr(low_products, lv & 0xFFFFu);
            const int wt = int(high >> 16) + int(lv >> 16);
            const uint32_t cand = ((high & 0xFFFFu) << 16) | (lv & 0xFFFFu);
            const bool hit = there && __fadd_rn(high_corr, lc) == target && (wt & 1) == cls &&
                             (even ? high_kap + half_kappa(nlo, lv) == kap : wt == w_total) && row_in_list(s, cls, wt, cand);
            const uint32_t any = __ballot_sync(0xFFFFFFFFu, hit);
            if (any) {
                row = __shfl_sync(0xFFFFFFFFu, cand, __ffs(int(any)) - 1);
                found = true;
            }
        }
    }
    // 3. its index: the shells of a class follow one another, rows of a shell ascend
    int wt = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) wt += rank_weight(int((row >> (4 * j)) & 7u));
    int begin = 0, end = 0;
    {
        constexpr int start[2][7] = {{0, 1, 29, 155, 499, 1256, 2048}, {0, 8, 72, 296, 808, 1816, 2048}};
        const int shell = wt >> 1;
#pragma unroll
        for (int q = 0; q < 6; ++q)
            if (shell == q) {
                begin = cls ? start[1][q] : start[0][q];
                end = cls ? start[1][q + 1] : start[0][q + 1];
            }
    }
    const uint32_t* rows = tab->paper.rows + 2048 * cls;
    const int stride = (end - begin + 31) >> 5;
    const int probe = begin + lane * stride;
    const uint32_t below = __ballot_sync(0xFFFFFFFFu, probe < end && __ldg(rows + (probe < end ? probe : 0)) <= row);
    const int block0 = begin + max(__popc(below) - 1, 0) * stride;
    const int at = block0 + lane;
    const uint32_t eq = __ballot_sync(0xFFFFFFFFu, lane < stride && at < end && __ldg(rows + (at < end ? at : 0)) == row);
    if (lane == 0) {
        S.found_row[s][e] = uint32_t(eq ? block0 + __ffs(int(eq)) - 1 : 0);
        S.found[s][e] = found && eq;
    }
}

// One warp: the winning entry of the objective, back through the join to the entries of the section tables.
__device__ __noinline__ void trace_join(EncShared& S, bool even, int end_pair, int par, int n) {
    const int lane = threadIdx.x & 31;
    const int cls3 = (even ? 0 : 1) ^ par;
    const int row_len = even ? kRow : kOddRow;
    const float *rows1[2] = {even ? S.F[0][0] : S.O[0][0], even ? S.F[0][1] : S.O[0][1]};
    const float *rows2[2] = {even ? S.F[1][0] : S.O[1][0], even ? S.F[1][1] : S.O[1][1]};
    const float* rows3 = even ? S.F[2][cls3] : S.O[2][cls3];
    const int gamma = end_pair & 7, xi = end_pair >> 3;
    // index after two sections and of the third
    int q = 0, k3 = 0;
    {
        const int j = lane, i = n - j;
        const int nb = even ? 10 : 6, na = even ? 19 : 10;
        const bool hit = j < nb && i >= 0 && i < na && __fadd_rn(S.win_H[i >= 0 && i < na ? i : 0], rows3[end_pair * row_len + (j < nb ? j : 0)]) == S.win_G;
        const uint32_t any = __ballot_sync(0xFFFFFFFFu, hit);
        if (any) {
            k3 = __ffs(int(any)) - 1;
            q = n - k3;
        }
    }
    // section 1's pair, class and index: lane = alpha + 8 c1 + 16 (half of the indices)
    const float h = S.win_H[q];
    const int alpha = lane & 7, c1 = (lane >> 3) & 1, c2 = c1 ^ par;
    const int p1 = alpha + 8 * xi, p2 = (alpha ^ gamma) + 8 * xi;
    const bool odd_end = odd_overlap(S.bytes[end_pair]) != 0;
    const int raised = even && !odd_end && odd_overlap(S.bytes[p1]) ? 1 : 0;
    const int shift = even ? 0 : (c1 & c2);
    int hit_i = -1;
    for (int i = lane >> 4; i < (even ? 11 : 6); i += 2) {
        const int j = q - shift - i;
        const int nb = even ? (c2 ? 8 : 9) : (c2 ? 4 : 5);
        if (hit_i < 0 && i >= raised && j >= 0 && j < nb &&
            __fadd_rn(rows1[c1][p1 * row_len + i - raised], rows2[c2][p2 * row_len + j]) == h)
            hit_i = i;
    }
    const uint32_t any = __ballot_sync(0xFFFFFFFFu, hit_i >= 0);
    const int src = any ? __ffs(int(any)) - 1 : 0;
    const int i1 = max(__shfl_sync(0xFFFFFFFFu, hit_i, src), 0);
    const int w_p1 = __shfl_sync(0xFFFFFFFFu, p1, src), w_p2 = __shfl_sync(0xFFFFFFFFu, p2, src);
    const int w_c1 = __shfl_sync(0xFFFFFFFFu, c1, src), w_c2 = w_c1 ^ par;
    const int w_raised = __shfl_sync(0xFFFFFFFFu, raised, src), w_shift = __shfl_sync(0xFFFFFFFFu, shift, src);
    const int j2 = max(q - w_shift - i1, 0);
    if (lane < 3) {
        const int pair = lane == 0 ? w_p1 : (lane == 1 ? w_p2 : end_pair), cls = lane == 0 ? w_c1 : (lane == 1 ? w_c2 : cls3);
        const int at = lane == 0 ? max(i1 - w_raised, 0) : (lane == 1 ? j2 : k3);
        const float* rows = lane == 0 ? rows1[w_c1] : (lane == 1 ? rows2[w_c2] : rows3);
        S.hit_pair[lane] = pair;
        S.hit_cls[lane] = cls;
        S.hit_k[lane] = at;
        S.hit_target[lane] = rows[pair * row_len + at];
    }
}

// Join and objective of one (end pair, class parity); keeps the better of this and what H, val, corr, arg hold.
template <bool EVEN, int PAR>
__device__ __forceinline__ void search_end(const EncShared& S, int end_pair, float (&H)[kH], float& val, float& corr, int& arg, int& par) {
    const bool odd_end = odd_overlap(S.bytes[end_pair]) != 0;
    const int m0 = EVEN ? (odd_end ? 1 : 0) : 2;  // squared norm = 16 (index + m0)
    float h[kH], v, c;
    int n;
    join_two<EVEN, PAR>(S, end_pair & 7, end_pair >> 3, odd_end, h);
    objective<EVEN, EVEN ? PAR : PAR ^ 1>(S, m0, end_pair, h, v, c, n);
    if (v > val) {
        val = v;
        corr = c;
        arg = n;
        par = PAR;
#pragma unroll
        for (int i = 0; i < kH; ++i) H[i] = h[i];
    }
}

// The file-order word (without the gain bit) of the traced winner; one warp.
__device__ __forceinline__ uint64_t winner_word(const EncShared& S, const DeviceTables* __restrict__ tab, bool even) {
    const int lane = threadIdx.x & 31;
    uint32_t c[3], row[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int e = S.found[s][0] ? 0 : 1;
        c[s] = S.bytes[S.hit_pair[s]] ^ (e ? 0xFFu : 0u);
        row[s] = S.found_row[s][e];
    }
    const uint32_t b1 = c[0] >> 7, b3 = c[2] >> 7, s8 = (b1 ? ~c[0] : c[0]) & 63u;
    const uint32_t leaves = tab->paper.branches[16 * s8 + (lane & 15)] & 0xFFu;
    const uint32_t eq = __ballot_sync(0xFFFFFFFFu, leaves == c[1]);
    const uint32_t b2 = eq ? uint32_t(__ffs(int(eq)) - 1) & 15u : 0u;
    const uint32_t i2 = row[1] + (S.hit_cls[1] ? uint32_t(kMiddleClass0) : 0u);
    return uint64_t(row[0]) | (uint64_t(i2) << 11) | (uint64_t(row[2]) << 22) | (uint64_t(s8) << 33) | (uint64_t(b1) << 39) |
           (uint64_t(b2) << 40) | (uint64_t(b3) << 44) | (uint64_t(even ? 0 : 1) << 45) | (uint64_t(uint32_t(S.hit_cls[0])) << 46);
}

__global__ void __launch_bounds__(kEncThreads * kEncGroups, 1)
k_encode(const float* __restrict__ w, const float* __restrict__ sigma, const DeviceTables* __restrict__ tab,
         unsigned char* __restrict__ codes, float* __restrict__ cosine, size_t nblocks) {
    extern __shared__ __align__(16) unsigned char enc_smem[];
    const int group = threadIdx.x / kEncThreads, tid = threadIdx.x - group * kEncThreads;
    EncShared& S = reinterpret_cast<EncShared*>(enc_smem)[group];
    if (tid < 64) S.bytes[tid] = uint8_t(pair_byte(tid));
    if (tid < 32) S.rs[tid] = tab->paper.rsqrt16m[tid];
    for (int i = tid; i < kHalfVectors; i += kEncThreads) S.halves[i] = kHalfList.v[i];
    if (tid <= kMaxW) S.low_index[tid] = kLowIndex.v[tid];
    const float gain0 = tab->gain[0], gain1 = tab->gain[1];

    // every group of every CTA takes the same number of turns; the first groups of all CTAs come first, so that few
    // blocks spread over all SMs
    const size_t per_turn = size_t(gridDim.x) * kEncGroups;
    const size_t place = size_t(group) * gridDim.x + blockIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    float next_w = 0.f;  // a turn ahead of its place in shared memory
    if (tid < 24) {
        S.w[0][tid] = place < nblocks ? w[place * 24 + tid] : 0.f;
        next_w = place + per_turn < nblocks ? w[(place + per_turn) * 24 + tid] : 0.f;
    }
    // The word of a traced block, its gain bit, its cosine; one warp.
    auto emit = [&](size_t block) {
        const bool live = S.out_live != 0;
        const float best_val = S.out_val;
        const uint64_t best_word = live && best_val > 0.f ? winner_word(S, tab, S.out_even != 0) : 0ull;
        if (block < nblocks && lane == 0) {
            const float sg_ = sigma ? sigma[block] : 1.f;
            // gain bit: argmin_g (gain sigma)^2 - 2 gain sigma <w, y> / |y|
            const float c = best_val;
            const float e0 = gain0 * sg_ * (gain0 * sg_ - 2.f * c), e1 = gain1 * sg_ * (gain1 * sg_ - 2.f * c);
            const uint64_t word = live ? best_word | (uint64_t(e1 < e0 ? 1u : 0u) << 47) : 0u;
#pragma unroll
            for (int k = 0; k < 6; ++k) codes[block * 6 + k] = uint8_t(word >> (8 * k));
            if (cosine) cosine[block] = live ? best_val / sqrtf(S.out_wn2) : 0.f;
        }
    };
    __syncthreads();
    int buf = 0;
    size_t first = 0;
    for (; first < nblocks; first += per_turn, buf ^= 1) {
        const size_t block = first + place;
        const float* w24 = S.w[buf];
        if (tid < 24) {
            S.w[buf ^ 1][tid] = next_w;
            next_w = block + 2 * per_turn < nblocks ? w[(block + 2 * per_turn) * 24 + tid] : 0.f;
        }
        float wn2 = 0.f;
#pragma unroll
        for (int j = 0; j < 24; ++j) wn2 = fmaf(w24[j], w24[j], wn2);
        const bool live = wn2 != 0.f;  // a zero block encodes as the all-zero word
        if (live) {
            // half tables, a thread per (section, nibble): warps 0 and 1 the high halves at even parity, 2 and 3 the low
            // ones, 4 and 5 the odd parity (warp 4 the outer sections, warp 5 the middle one)
            const int nibble = tid & 15;
            if (tid < 128) {
                const int s = (tid & 63) >> 4;
                if (s < 3) {
                    if (tid < 64) half_even<true>(w24 + 8 * s + 4, nibble, s == 1, S.hi[s] + nibble * kHiStride);
                    else half_even<false>(w24 + 8 * s, nibble, s == 1, S.lo[s] + nibble * kLoStride);
                }
            } else if (tid < 160) {
                const int s = (tid & 16) ? 2 : 0;
                half_odd<true, false>(w24 + 8 * s + 4, nibble, S.hi_odd[s] + nibble * kOddHiStride);
                half_odd<false, false>(w24 + 8 * s, nibble, S.lo_odd[s] + nibble * kOddLoStride);
            } else if ((tid & 16) == 0) {
                half_odd<true, true>(w24 + 12, nibble, S.hi_odd[1] + nibble * kOddHiStride);
                half_odd<false, true>(w24 + 8, nibble, S.lo_odd[1] + nibble * kOddLoStride);
            }
        }
        if (warp == 5 && first) emit(block - per_turn);  // the block of the turn before; this warp's half tables are the shortest
        __syncthreads();
        if (live) {  // section tables at even parity, two warps per section; the schedulers of warps 0 and 1 have a warp more
                     // than the others and get the middle section's, the shorter ones
            const int pair = tid & 63;
            if (tid < 64) section_rows<true, true>(S, 1, pair);
            else section_rows<true, false>(S, tid < 128 ? 0 : 2, pair);
        }
        __syncthreads();
        // Join and objective.  Even parity: warps 0..3, thread = (end pair, class parity).  The odd parity has rows of
        // six entries instead of ten and eleven: warps 4 and 5 do its section tables and both class parities meanwhile.
        float H[kH];
        float val = kNeg, corr = kNeg;
        int arg = 0, par = 0;
        if (live) {
            if (warp < 4) {
                if (warp < 2) search_end<true, 0>(S, tid & 63, H, val, corr, arg, par);
                else search_end<true, 1>(S, tid & 63, H, val, corr, arg, par);
            } else {
                const int pair = tid - 128;
                section_rows<false, false>(S, 0, pair);
                section_rows<false, true>(S, 1, pair);
                section_rows<false, false>(S, 2, pair);
                asm volatile("bar.sync %0, 64;" ::"r"(1 + group) : "memory");
                search_end<false, 0>(S, pair, H, val, corr, arg, par);
                search_end<false, 1>(S, pair, H, val, corr, arg, par);
            }
            // the warp's best; the objective of a non-zero block is positive at its best, so bit patterns compare like values
            const uint32_t bits = val > 0.f ? __float_as_uint(val) : 0u;
            const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, bits);
            const uint32_t who = __ballot_sync(0xFFFFFFFFu, bits == top);
            if (lane == __ffs(int(who)) - 1) {
                S.red_val[warp] = top ? val : kNeg;
                S.red_arg[warp] = uint32_t(tid);
            }
        }
        __syncthreads();
        float best_val = kNeg;
        uint32_t winner = 0;
        if (live) {  // the odd parity first: it keeps ties
            best_val = S.red_val[4];
            winner = S.red_arg[4];
#pragma unroll
            for (int k = 5; k < 10; ++k)
                if (S.red_val[k % 6] > best_val) {
                    best_val = S.red_val[k % 6];
                    winner = S.red_arg[k % 6];
                }
        }
        const bool best_even = winner < 128u;
        if (uint32_t(warp) == winner >> 5) {  // the winner's warp traces it through the join
            if (live && best_val > 0.f) {
                if (uint32_t(tid) == winner) {
#pragma unroll
                    for (int i = 0; i < kH; ++i) S.win_H[i] = H[i];
                    S.win_G = corr;
                    S.win_arg = arg;
                    S.win_par = par;
                }
                __syncwarp();
                trace_join(S, best_even, int(winner) & 63, S.win_par, S.win_arg);
            } else if (lane < 3) {
                S.hit_pair[lane] = S.hit_cls[lane] = S.hit_k[lane] = 0;  // what a block without a best point (NaN) is traced to
            }
        }
        __syncthreads();
        if (live) {  // a warp per section and byte of its pair
            trace_section(S, tab, w24, best_even, warp >> 1, warp & 1);
        }
        if (tid == 160) {
            S.out_val = best_val;
            S.out_wn2 = wn2;
            S.out_live = live;
            S.out_even = best_even;
        }
        __syncthreads();
    }
    if (warp == 5) emit(first - per_turn + place);
}

}  // namespace

cudaError_t launch_encode(const float* w, const float* sigma, const void* table, unsigned char* codes, float* cosine,
                          size_t nblocks, cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const int smem = int(sizeof(EncShared)) * kEncGroups;
    static PerDeviceOnce once;
    e = once.run([smem] { return cudaFuncSetAttribute(k_encode, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
    if (e != cudaSuccess) return e;
    const unsigned grid = unsigned(nblocks < size_t(sms) ? nblocks : size_t(sms));
    k_encode<<<grid, kEncThreads * kEncGroups, smem, s>>>(w, sigma, static_cast<const DeviceTables*>(table), codes, cosine, nblocks);
    return cudaGetLastError();
}

}  // namespace tetra
