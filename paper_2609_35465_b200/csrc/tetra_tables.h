// Host-side construction of the Tetra decode tables (Sec. 3.2-3.4) and of the
// derived lookup tables the sm_100a kernels stage in shared memory.
#pragma once
#include <cstddef>
#include <cstdint>

namespace tetra {

// The tables exactly as the paper lays them out (Sec. 3.4): 18,816 bytes.
struct PaperTables {
    uint32_t rows[4096];      // rank rows, class 0 then class 1, nibble j = rank of coordinate j
    uint8_t prefixes[128];    // [2*s8 + b1]
    uint16_t branches[1024];  // [16*s8 + b2] = middle byte | s16 << 8
    uint8_t suffixes[128];    // [2*s16 + b3]
    float rsqrt16m[32];       // 1/sqrt(16 m), entry 0 = 0
};
static_assert(sizeof(PaperTables) == 18816, "paper table blob is 18,816 bytes");

constexpr uint32_t kTableMagic = 0x54455442u;  // "TETB"
constexpr uint32_t kTableVersion = 11;
// Nibble of a fast table word that belongs to coordinate j of a section: neighbours are sixteen bits apart, so that one
// mask picks the pair (j, j + 1) as the two halves of a register.
constexpr int fast_nibble(int j) { return (j >> 1) + 4 * (j & 1); }
constexpr int kMiddleClass0 = 1240;            // N0 of Sec. 3.3 (checked at build)
// The last row of a class's 2048 and of the middle list's class 0 (checked at build): each cuts a shell of equal
// cost at this packed value; the middle list's class 1 ends with a whole shell.
constexpr uint32_t kLastRowClass0 = 0x11030011u, kLastRowClass1 = 0x00222011u, kLastRowMiddle0 = 0x30001010u;

// Everything tetra_build_table copies to the device, in one blob.
struct DeviceTables {
    PaperTables paper;          //     0: file-order decode (tetra_decode_blocks, paper-design GEMV)
    float gain[2];              // 18816
    uint32_t magic;             // 18824
    uint32_t version;           // 18828
    // ---- fast path: everything below is staged in shared memory ------------
    // Rank rows, class by class: nibble fast_nibble(j) = -2 k (two's complement) of coordinate j's rank,
    // k = 0, 1, -1, 2, -2.
    // (the kernels place this part on a 16 KiB boundary of shared memory, so each
    //  sub-table's offset can be OR-ed into an index instead of added)
    uint32_t rows_fast[4096];   // +0
    uint32_t mid_fast[2048];    // +16384: rows_fast[mix(i2)], indexed by i2 directly
    float scale[32][2];         // +24576: -gain[0] / sqrt(16 m) in entry [m][0], 8 bytes per m: sixteen neighbouring norms in
                                //         different banks.  Minus: the fast decoder emits minus (eight times) the point.
    // Pattern-byte masks of the Turyn coordinates: nibble fast_nibble(j) all ones where the Hamming word has coordinate j
    // set; H for a and b, H' for x.  mask_xp has x and the parity in one index, x << 1 | p, and is complemented
    // where p = 1.
    uint32_t mask_h[16];        // +24832
    uint32_t spare0_[16];       // +24896
    uint32_t mask_xp[32];       // +24960
    uint32_t spare1_[128];      // +25088
    float scale1[32][2];        // +25600: the same for gain[1], at a power of two from the first
    // ---- pack-time only (global memory) ------------------------------------
    // 12 trellis bits (s8 | b1<<6 | b2<<7 | b3<<11) -> Turyn coordinates a | b<<4 | x<<8.
    uint16_t trellis_to_abx[4096];
    uint32_t spare2_[320];      // the blob keeps its size
};

constexpr size_t kFastOffset = offsetof(DeviceTables, rows_fast);
constexpr size_t kFastBytes = offsetof(DeviceTables, trellis_to_abx) - kFastOffset;
static_assert(kFastOffset % 16 == 0 && kFastBytes % 16 == 0, "staged part must be 16-byte copyable");

// Fills `out` (gain from gain2, or the defaults when null).  Returns 0, or a
// negative number naming the structural check that failed (never expected).
int build_device_tables(DeviceTables* out, const float* gain2);

// The two scale tables from the gains and rsqrt16m.
void fill_scales(DeviceTables* t);

}  // namespace tetra
