// Decode-and-multiply for 2..16 activation vectors at once (Eq. (2), Sec. 5.1): a block is decoded once and
// multiplied with every vector, in one launch.
//
// The products of a block's 24 coordinates with up to 16 vectors are a small dense contraction and run on the tensor
// cores: mma.sync m16n8k16, float16 x float16 with float32 accumulation.  Half of minus a coordinate, -y / 2 = z + p / 2,
// is a float16 that two logic operations and one addition make from the decoder's nibbles, and the activations ARE
// float16, so both operands and every product are exact.  (The three int8 planes of 24-bit fixed point that the batch-1
// kernels use cost three times the MMAs and five instructions per result here; the float32 result costs half a packed
// FFMA.)  mma.sync rather than tcgen05: a CTA owns about 28 rows of a 4096-row matrix, a tile of 16 rows keeps sixteen
// warps busy with that, 128 rows would not.
//
// Lane 4 q + t decodes rows 2 q and 2 q + 1 of a 16-row tile at column t of four.  Two ways from there:
//   up to four vectors: straight from registers.  An MMA takes four coordinates of both blocks from every lane as A
//   (rows q and q + 8), and B is block diagonal -- column 2 t + v of B is zero outside the k range that lane t feeds --
//   so D[q][2 t + v] is the product of lane (q, t)'s own block with vector v of its own column and arrives in that same
//   lane, next to the block's scale: six MMAs for two blocks per lane and two vectors, no shuffle, no shared-memory
//   tile, and B is the activations as they lie in memory (rows that are not 16-byte aligned: shifted to where aligned ones are);
//   five and more: dense B.  A block's 24 halves go through a shared-memory tile whose rows keep stores and ldmatrix
//   conflict-free, an MMA pair (k16 + k8) multiplies sixteen blocks of ONE column with eight vectors, and the
//   block's scale reaches the lanes that hold its results by a shuffle.
// The line lies where the tensor pipe's time for the zeros overtakes the tile.  Block diagonal / dense, 2, 3, 4 vectors:
// 4096 x 4096 7.1 / 9.0, 8.2 / 9.1, 8.2 / 9.2 us; 4096 x 12288 12.8 / 18.6, 15.5 / 18.7, 15.7 / 18.9; 1024 x 4096
// 4.0 / 4.9, 4.5 / 4.9, 4.5 / 4.9.  Eight and sixteen on 4096 x 4096, in an earlier series: 9.3 and 13.3 us in a build that
// had them block diagonal, 8.7 and 10.1 dense.  (Int8 planes, activations staged by the CTA and a combining kernel: 13.5 us
// for three vectors on 4096 x 4096, 27.8 us for sixteen on 4096 x 12288, against 7.7 and 22.1.)
//
// A warp's step is NT row tiles x four block columns.  The sixteen warps of a CTA take every sixteenth column quad, so a
// warp needs nothing from the others until the end: its words come straight from global memory one step ahead, the four
// columns' activations through its own cp.async buffer, and its accumulators live in registers.
//
// One launch, no scratch memory: what a call of a few microseconds consists of is latency, and a second kernel that
// adds the CTAs' partial sums costs more than the products of a 4096 x 4096 matrix.  A CTA owns whole rows; where
// rows are too few for all SMs, a cluster of two CTAs shares them, each takes a range of columns, and the partial sums
// meet through distributed shared memory.  Sums are added in warp order, then CTA order: bit-identical from run to run.
//
// Bound by instruction issue in the steps (decode and conversion) and, for small matrices, by the chain of launch,
// tables, one step and sums.
#include <cuda_fp16.h>

#include "q4_common.cuh"
#include "tetra_gemv_common.cuh"
#include "tetra_rows.h"

namespace tetra {

constexpr uint32_t kXVec = 4 * 48 + 16;        // bytes per vector of an activation buffer: four columns, and a line of zeros
                                               // or what a row that is not aligned needs more
constexpr int kBatMaxTiles = 4;                // row tiles of a step

struct BatParams {
    const unsigned char* codes;
    const float* row_scales;
    const __half* x;
    const __half* tail;
    float* y;
    int32_t N, K, B, batch;
    int32_t tiles, quads;    // row tiles of 16, column quads
    int32_t groups;          // clusters: groups of CTAs that share rows
    int32_t cluster;         // CTAs of a cluster
};

constexpr int kBatWarps = 16, kBatThreads = 32 * kBatWarps;
constexpr uint32_t kTileCol = 16 * 48 + 32;    // bytes per column of a shared-memory tile: 16 rows of 24 halves, bank spread
constexpr uint32_t kTileBytes = 4 * kTileCol;  // four columns

// G: vector pairs (block diagonal) or groups of eight (dense); slots: vectors they make room for.
constexpr int bat_slots(bool dense, int g) { return (dense ? 8 : 2) * g; }
// Dense: tiles decoded together.  Four blocks in flight per lane hide the table lookups better than two; with two
// groups the registers do not allow it.
constexpr int bat_together(bool dense, int g, int nt) { return dense && g == 1 && nt > 1 ? 2 : 1; }
// Activation buffers of a warp.  Dense: the fragments of a step's columns go to registers at its start, once for all its
// tiles, so one buffer serves (read per tile they were a sixth of the shared-memory traffic, which keeps its pipe 78 %
// busy: 4096 x 12288, 16 vectors 2 us more).
constexpr bool bat_hold(bool dense) { return dense; }
// Block diagonal: two by turns, or, for rows of x that are not aligned, one for them as they lie in memory and one for
// them in their places: it is filled at the start of a step, when the step before has been read.
constexpr uint32_t bat_buffers(bool dense) { return bat_hold(dense) ? 1 : 2; }
// Whether a step asks for the next quad's activations behind its first tile's lookups instead of ahead of them.  Ahead /
// behind, us, two vectors: one tile 2048 x 2304 3.47 / 3.54 (700 x 800 2.23 / 2.19), two tiles 4096 x 12288 13.5 / 12.7, three
// 5003 x 7008 12.3 / 11.8, four 9000 x 1104 4.79 / 4.73.  Four vectors gain with two tiles only (4096 x 12288 15.6 / 15.1, but
// 9728 x 2560 13.6 / 13.8 and 2048 x 2304 3.83 / 3.87) and stay ahead.  Rows that are not aligned are put into their places
// there too: two tiles, 4096 x 4097 with 2 / 3 vectors, 7.8 / 9.2 ahead and 7.5 / 9.1 behind; one, 700 x 804 with three, 2.95
// and 3.00; four, 9000 x 1100 with three, 6.6 and 7.1.
constexpr bool bat_late(bool dense, int g, int nt, bool wide) { return !dense && (wide ? g == 1 && nt > 1 : nt == 2); }
// Row stride, in floats, of the partial sums: even, so that pairs stay aligned.
constexpr int bat_stride(bool dense, int g) { return bat_slots(dense, g) + 2; }
struct BatSmem {
    // offsets from the 16 KiB-aligned table copy; total includes the alignment slack.  A warp's area: its activation
    // buffers, then its tiles (dense); the partial sums of all warps take the areas' place at the end.
    uint32_t warps, per_warp, rs, tail, xtail, total;
};
constexpr BatSmem bat_smem(bool dense, int g, int nt) {
    BatSmem S{};
    S.warps = uint32_t(kFastBytes);
    S.per_warp = bat_buffers(dense) * uint32_t(bat_slots(dense, g)) * kXVec + (dense ? uint32_t(bat_together(dense, g, nt)) * kTileBytes : 0u);
    const uint32_t sums = uint32_t(nt * 16 * bat_stride(dense, g) * 4);  // per warp
    S.rs = S.warps + kBatWarps * (S.per_warp > sums ? S.per_warp : sums);
    S.tail = S.rs + uint32_t(nt) * 64u;                 // half [rows][24]
    S.xtail = S.tail + uint32_t(nt) * (16u * 48u);      // float [16][24]
    S.total = S.xtail + 16u * 96u + kSmAlign;
    return S;
}
static_assert(bat_smem(false, 2, 4).total <= 227 * 1024 && bat_smem(true, 1, 4).total <= 227 * 1024 &&
              bat_smem(true, 2, 4).total <= 227 * 1024, "shared memory");
template <bool DENSE, int G, int NT, bool WIDE>
struct BatShape {
    static constexpr int slots = bat_slots(DENSE, G), together = bat_together(DENSE, G, NT), stride = bat_stride(DENSE, G);
    static constexpr bool hold = bat_hold(DENSE);
    static constexpr uint32_t buffers = bat_buffers(DENSE);
    static constexpr bool late = bat_late(DENSE, G, NT, WIDE);
    static constexpr BatSmem smem = bat_smem(DENSE, G, NT);
};

// Half of minus the point, float16 x 2: a[4 s + t] = coordinates 2 t and 2 t + 1 of section s.  Returns the block's scale
// (minus the gain over sqrt(16 m)).  A nibble z sits in the mantissa of 64 (as z + 8: the exclusive or that sets
// the exponent flips its sign bit) with p in the bit below: 72 + z + p / 2.  The squared norm of the halves, 4 m, is
// exact in float16 (at most 104, terms of a quarter); with 1024 added it is the mantissa itself.
template <bool HI>
__device__ __forceinline__ float decode_halves(uint32_t sm_tab, uint32_t w0, uint32_t w1pair, uint32_t (&a)[12]) {
    NibbleBlock nb;
    decode_nibbles<HI>(sm_tab, w0, w1pair, nb);
    const uint32_t magic = (nb.p4 & 4u) * 0x00020002u + 0x54805480u;
    const __half2 bias = __half2half2(__ushort_as_half(0xD480));  // -72
    __half2 n0{}, n1{};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const uint32_t z = nb.z[s];
        const uint32_t v[4] = {((z << 4) & 0x00F000F0u) ^ magic, (z & 0x00F000F0u) ^ magic, ((z >> 4) & 0x00F000F0u) ^ magic,
                               ((z >> 8) & 0x00F000F0u) ^ magic};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const __half2 h = __hadd2(*reinterpret_cast<const __half2*>(&v[t]), bias);
            a[4 * s + t] = *reinterpret_cast<const uint32_t*>(&h);
            __half2& n = (t & 1) ? n1 : n0;
            n = (s == 0 && t < 2) ? __hmul2(h, h) : __hfma2(h, h, n);
        }
    }
    const __half2 n = __hadd2(n0, n1);
    const __half m4 = __hadd(__hadd(__low2half(n), __high2half(n)), __ushort_as_half(0x6400));  // 1024 + 4 m
    return lds32f(uint32_t(__half_as_ushort(m4)) * 2u + (nb.norm0 >> kNormShift) - 0x6400u * 2u);
}

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float cluster_load(uint32_t saddr, uint32_t rank) {
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(saddr), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

// DENSE, G: see bat_slots; NT: row tiles of a step; WIDE: every row of x is 16-byte aligned.
template <bool DENSE, int G, int NT, bool WIDE>
__global__ void __launch_bounds__(kBatThreads, 1)
k_gemv_batched(const DeviceTables* __restrict__ tab, const __grid_constant__ BatParams P) {
    using Shape = BatShape<DENSE, G, NT, WIDE>;
    constexpr int PS = Shape::stride, W = kBatWarps, THREADS = kBatThreads, SLOTS = Shape::slots, TW = Shape::together;
    constexpr BatSmem S = Shape::smem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_release();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = lane >> 2, t = lane & 3;
    const int V = SLOTS == 2 ? 2 : P.batch, C = P.cluster;  // one vector takes another kernel
    const int group = int(blockIdx.x) / C, rank = int(blockIdx.x) - group * C;
    // this CTA's row tiles (shared with its cluster) and column quads
    const int tile_lo = int((long long)group * P.tiles / P.groups), tile_hi = int((long long)(group + 1) * P.tiles / P.groups);
    const int quad_lo = rank * P.quads / C, quad_hi = (rank + 1) * P.quads / C;
    const uint32_t sm_raw = smem_u32(smem_raw);
    unsigned char* smem = smem_raw + (((sm_raw + kSmAlign - 1) & ~(kSmAlign - 1)) - sm_raw);
    const uint32_t sm_tab = smem_u32(smem);
    float* part = reinterpret_cast<float*>(smem + S.warps);
    float* rs_sm = reinterpret_cast<float*>(smem + S.rs);
    __half* tail_sm = reinterpret_cast<__half*>(smem + S.tail);
    float* xtail = reinterpret_cast<float*>(smem + S.xtail);
    constexpr uint32_t kXBuf = SLOTS * kXVec;
    const uint32_t xbuf = sm_tab + S.warps + uint32_t(warp) * S.per_warp;
    [[maybe_unused]] const uint32_t tile = xbuf + Shape::buffers * kXBuf;
    const int ntail = P.tail ? P.K % 24 : 0, Kx = min(P.K, 24 * P.B);

    // This lane's words of a step: rows 2 q and 2 q + 1 of NT tiles at column t.  Rows and columns outside the matrix
    // repeat a row group or column inside: such rows are not stored, such columns meet zeros.  words_at moves the
    // lane's address to a quad; a tile is a uniform offset from there.
    uint2 w0[NT];
    uint32_t w1[NT];
    const int last_rg = (P.N + 7) / 8 - 1;
    const unsigned char* words = nullptr;
    const uint32_t lane_w0 = uint32_t((q >> 1) & 1) * uint32_t(P.B) * 16u + uint32_t(q & 1) * 8u;
    const uint32_t lane_w1 = uint32_t(2 * P.B) * 16u + uint32_t(q & 3) * 4u;
    auto words_at = [&](int t0, int quad) {
        words = P.codes + (size_t(min(2 * t0 + (q >> 2), last_rg)) * 3 * P.B + min(4 * quad + t, P.B - 1)) * 16;
    };
    auto load_words = [&](int i, int t0) {
        const int up = min(2 * i, max((last_rg - 2 * t0 - (q >> 2)) & ~1, 0));  // row groups from the first tile's
        const unsigned char* at = words + uint32_t(up) * 48u * uint32_t(P.B);
        w0[i] = __ldg(reinterpret_cast<const uint2*>(at + lane_w0));
        w1[i] = __ldg(reinterpret_cast<const uint32_t*>(at + lane_w1));
    };
    auto stage_rows = [&](int t0, int nt) {
        const int row0 = 16 * t0, rows = min(16 * nt, P.N - row0);
        for (int i = threadIdx.x; i < rows; i += THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(smem_u32(rs_sm + i)), "l"(P.row_scales + row0 + i));
        if (ntail) {
            const __half* tl = P.tail + size_t(row0) * ntail;
            for (int r = threadIdx.x >> 3; r < rows; r += THREADS / 8)
                for (int k = threadIdx.x & 7; k < ntail; k += 8) tail_sm[r * 24 + k] = tl[size_t(r) * ntail + k];
        }
    };
    // The activations of a quad's four columns, twelve units of eight per vector, into buffer `slot`; zeros beyond the
    // last column.  Lanes 0..23: unit lane % 12 of every second vector.
    const int x_v = lane >= 12 ? 1 : 0, x_u = lane - 12 * x_v;
    // How addresses and tests are written moves the registers of the loops behind, and the time by 1 to 3 %.  Best of those
    // tried: offsets from x for four vectors (pointers: 5003 x 7008 with three 13.85 us, offsets 13.46), pointers elsewhere;
    // one test for lane and vector with eight copies (5003 x 7008 with 11 vectors: two tests 18.85, one 18.65).
    [[maybe_unused]] const __half* x_src = P.x + size_t(x_v) * P.K + 8 * x_u;
    [[maybe_unused]] const uint32_t x_off = uint32_t(x_v) * uint32_t(P.K) + 8u * uint32_t(x_u);
    [[maybe_unused]] const int x_left = Kx - 8 * x_u;
    [[maybe_unused]] const int x_first = SLOTS == 16 && lane >= 24 ? SLOTS : x_v;
    [[maybe_unused]] auto stage_aligned = [&](uint32_t slot, int quad) {
        const int k = 96 * quad;
        const uint32_t dst = xbuf + slot * kXBuf + uint32_t(x_v) * kXVec + uint32_t(x_u) * 16u;
        auto copy = [&](int i, const __half* src, int n) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" :: "r"(dst + uint32_t(i) * 2u * kXVec), "l"(src), "r"(2 * n));
        };
        if constexpr (SLOTS == 4) {
            const int n = min(max(x_left - k, 0), 8);
#pragma unroll
            for (int i = 0; i < SLOTS / 2; ++i)
                if (lane < 24 && 2 * i + x_v < V) copy(i, P.x + (n ? x_off + uint32_t(k) + uint32_t(2 * i) * uint32_t(P.K) : 0u), n);
        } else {
            const int n = min(max(Kx - 8 * x_u - k, 0), 8);
            const __half* src = n ? x_src + k : P.x;
            const size_t step = n ? 2 * size_t(P.K) : 0;
#pragma unroll
            for (int i = 0; i < SLOTS / 2; ++i, src += step)
                if ((SLOTS == 16 || lane < 24) && 2 * i + x_first < V) copy(i, src, n);
        }
    };
    // Rows of x that are not 16-byte aligned come as they lie in memory, thirteen aligned units: a vector's quad starts
    // x_skip halves into its part of the buffer, the same for all quads.  What the first unit brings along from ahead of
    // the row is not used.  (Loaded, shifted and stored by the lanes, a pair of vectors after the other, a step waited for
    // memory up to eight times.  5003 x 7001 with 2 / 3 / 8 / 16 vectors 13.7 / 17.6 / 24.9 / 37.3 us, 13.4 / 16.4 / 20.1 / 25.5
    // this way.  Two vectors are up to 3 % slower where a warp has a step or two, 2048 x 2305 4.03 and 4.09: a step more of
    // shared memory in a short chain.)
    [[maybe_unused]] constexpr uint32_t kRaw = Shape::hold ? 0u : 1u;  // dense: the fragments are read from where the rows arrive
    const uint32_t x_half = uint32_t(reinterpret_cast<uintptr_t>(P.x) >> 1);
    [[maybe_unused]] auto x_skip = [&](int v) { return row_skip(x_half, v, P.K); };
    [[maybe_unused]] const __half* x_unit = P.x + (8u - x_skip(0));  // an aligned address, for copies of nothing
    [[maybe_unused]] auto stage_raw = [&](int quad, int first_unit) {
        const int v0 = lane >= kRowUnits ? 1 : 0, u = lane - kRowUnits * v0;
        auto copy = [&](int v) {
            const RowUnit unit = row_unit(x_skip(v), quad, u, Kx);
            const __half* src = P.x + (ptrdiff_t(v) * P.K + unit.from);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" :: "r"(xbuf + kRaw * kXBuf + uint32_t(v) * kXVec + uint32_t(u) * 16u),
                         "l"(unit.halves ? src : x_unit), "r"(2 * unit.halves));
        };
        if constexpr (DENSE || NT == 1) {  // a loop is less code ahead of a short launch's only step: 700 x 804 with four vectors 2.80 us, unrolled 2.95
            if (u >= first_unit && u < kRowUnits)
#pragma unroll 2
                for (int v = v0; v < V; v += 2) copy(v);
        } else {
#pragma unroll
            for (int i = 0; i < SLOTS / 2; ++i)
                if (u >= first_unit && u < kRowUnits && 2 * i + v0 < V) copy(2 * i + v0);
        }
    };
    // Quad 0 of rows that begin within a unit: the first units half by half, for nothing is read ahead of x.
    [[maybe_unused]] auto stage_raw_begin = [&] {
        constexpr int PER = (SLOTS * 8 + 31) / 32;
        unsigned short begin[PER];
        const int h = lane & 7;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int v = 4 * i + (lane >> 3), k = h - int(x_skip(v));
            begin[i] = v < V && k >= 0 && k < Kx ? __half_as_ushort(P.x[size_t(v) * P.K + k]) : (unsigned short)0;
        }
        stage_raw(0, 1);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int v = 4 * i + (lane >> 3);
            if (v < V)  // zeros ahead of the row: not used
                asm volatile("st.shared.u16 [%0], %1;" :: "r"(xbuf + kRaw * kXBuf + uint32_t(v) * kXVec + 2u * uint32_t(h)), "h"(begin[i]) : "memory");
        }
    };
    auto stage_x = [&](uint32_t slot, int quad) {
        if constexpr (WIDE) stage_aligned(slot, quad);
        else stage_raw(quad, 0);
    };
    // 32 bits that start `skip` halves on from a word of shared memory
    [[maybe_unused]] auto lds_from = [&](uint32_t at, uint32_t skip) {
        uint32_t lo, hi;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(lo) : "r"(at + 4u * (skip >> 1)));
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(hi) : "r"(at + 4u * (skip >> 1) + 4u));
        return __funnelshift_r(lo, hi, 16u * (skip & 1u));
    };

    // ---- before the wait: what does not depend on the activations ------------------------------------------
    if (quad_lo + warp < quad_hi) {
        words_at(tile_lo, quad_lo + warp);
#pragma unroll
        for (int i = 0; i < NT; ++i) load_words(i, tile_lo);
    }
    stage_fast_tables_async(tab, smem_raw);
    stage_rows(tile_lo, min(tile_hi - tile_lo, NT));
    pdl_wait();  // x may come from the preceding kernel
    for (int i = threadIdx.x; i < V * 24; i += THREADS) {
        const int v = i / 24, k = i - 24 * v;
        xtail[i] = k < ntail ? __half2float(P.x[size_t(v) * P.K + 24 * P.B + k]) : 0.f;
    }

    // Block diagonal: lane 4 q + t holds its column of B's coordinates only where q / 2 = t, of vector q % 2 of a pair;
    // the other lanes (and a vector beyond the last) read a line of zeros.  Dense: word t of a section, of vector q of
    // a group (results beyond the last vector are never used, whatever they are).
    const bool mine = (q >> 1) == t;
    [[maybe_unused]] const bool x_words = WIDE || ((reinterpret_cast<uintptr_t>(P.x) | (uintptr_t(P.K) * 2)) & 3) == 0;  // fragments are words of the buffer
    uint32_t x_lane[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (DENSE) x_lane[g] = uint32_t(min(8 * g + q, V - 1)) * kXVec + uint32_t(t) * 4u + (!WIDE && x_words ? 2u * x_skip(min(8 * g + q, V - 1)) : 0u);
        else x_lane[g] = mine && 2 * g + (q & 1) < V ? uint32_t(2 * g + (q & 1)) * kXVec + uint32_t(t) * 48u : 192u;
    }
    const uint32_t x_step = mine ? 16u : 0u;

    for (int t0 = tile_lo; t0 < tile_hi; t0 += NT) {
        const int nt = min(tile_hi - t0, NT);
        // rows 2 q (k = 0, 1) and 2 q + 1 (k = 2, 3): block diagonal, the lane's own column, vectors 2 g and 2 g + 1;
        // dense, all columns, vectors 8 g + 2 t and 8 g + 2 t + 1
        float acc[NT][G][4];
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[i][g][k] = 0.f;
        if (t0 != tile_lo) {
            __syncthreads();  // the sums of the tiles before have been read
            stage_rows(t0, nt);
            if (quad_lo + warp < quad_hi) {
                words_at(t0, quad_lo + warp);
#pragma unroll
                for (int i = 0; i < NT; ++i) load_words(i, t0);
            }
        }
        uint32_t slot = 0;
        if (!WIDE && quad_lo + warp == 0 && rows_begin_within_a_unit(x_half)) stage_raw_begin();
        else if (quad_lo + warp < quad_hi) stage_x(0, quad_lo + warp);
        if (!DENSE && lane < (WIDE ? 2 : 1))  // the line of zeros in the buffers that fragments are read from
            asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" :: "r"(xbuf + uint32_t(lane) * kXBuf + 192u), "r"(0u) : "memory");
        asm volatile("cp.async.commit_group;");
        if (t0 == tile_lo) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();  // the tables are in place
        }
        for (int quad = quad_lo + warp; quad < quad_hi; quad += W) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();  // every lane's copies have landed, and every lane has left the other buffer
            const int next = min(quad + W, quad_hi - 1);
            const uint32_t x_at = xbuf + slot * kXBuf;
            [[maybe_unused]] uint32_t b_held[4][G][3];
            if constexpr (Shape::hold) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int s = 0; s < 3; ++s) {
                            const uint32_t from = x_at + x_lane[g] + uint32_t(48 * j + 16 * s);
                            if (x_words) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b_held[j][g][s]) : "r"(from));
                            else b_held[j][g][s] = lds_from(from, x_skip(min(8 * g + q, V - 1)));
                        }
                __syncwarp();
            }
            auto stage_next = [&] {
                if constexpr (!Shape::hold && !WIDE) {  // into their places, a lane a word; the next rows then take the ones in memory order
#pragma unroll
                    for (int i = 0; i < SLOTS * 48 / 32; ++i) {
                        const int id = lane + 32 * i, v = id / 48, word = id - 48 * v;
                        if (v < V)
                            asm volatile("st.shared.u32 [%0], %1;" :: "r"(x_at + uint32_t(v) * kXVec + 4u * uint32_t(word)),
                                         "r"(lds_from(xbuf + kRaw * kXBuf + uint32_t(v) * kXVec + 4u * uint32_t(word), x_skip(v))) : "memory");
                    }
                    __syncwarp();
                }
                if (quad + W < quad_hi) stage_x(Shape::hold ? 0u : slot ^ 1u, next);
                asm volatile("cp.async.commit_group;");
            };
            if constexpr (!Shape::late) stage_next();
            words_at(t0, next);
            if constexpr (!DENSE) {
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    uint32_t a[2][12];
                    const float s0 = decode_halves<false>(sm_tab, w0[i].x, w1[i], a[0]);
                    const float s1 = decode_halves<true>(sm_tab, w0[i].y, w1[i], a[1]);
                    load_words(i, t0);
                    if (Shape::late && i == 0) stage_next();
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int m = 0; m < 3; ++m) {
                            uint32_t b[4];
                            q4_lds128(x_at + x_lane[g] + m * x_step, b);
                            const uint32_t a0[4] = {a[0][4 * m], a[1][4 * m], a[0][4 * m + 1], a[1][4 * m + 1]};
                            const uint32_t a1[4] = {a[0][4 * m + 2], a[1][4 * m + 2], a[0][4 * m + 3], a[1][4 * m + 3]};
                            mma_k16(d, a0, b[0], b[1]);
                            mma_k16(d, a1, b[2], b[3]);
                        }
                        fma2(s0, d[0], d[1], acc[i][g][0], acc[i][g][1]);
                        fma2(s1, d[2], d[3], acc[i][g][2], acc[i][g][3]);
                    }
                }
            } else {
#pragma unroll
                for (int i0 = 0; i0 < NT; i0 += TW) {
                    constexpr int kLeft = NT % TW;  // an odd last tile goes alone
                    const int tw = i0 + TW <= NT ? TW : kLeft;
                    float scale[TW][2];
#pragma unroll
                    for (int k = 0; k < tw; ++k) {
                        const int i = i0 + k;
#pragma unroll
                        for (int rg = 0; rg < 2; ++rg) {
                            uint32_t a[12];
                            scale[k][rg] = rg ? decode_halves<true>(sm_tab, w0[i].y, w1[i], a) : decode_halves<false>(sm_tab, w0[i].x, w1[i], a);
                            const uint32_t dst = tile + uint32_t(k) * kTileBytes + uint32_t(t) * kTileCol + uint32_t(8 * rg + q) * 48u;
#pragma unroll
                            for (int s = 0; s < 3; ++s)
                                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" :: "r"(dst + 16u * s), "r"(a[4 * s]), "r"(a[4 * s + 1]),
                                             "r"(a[4 * s + 2]), "r"(a[4 * s + 3]) : "memory");
                        }
                        load_words(i, t0);
                    }
                    __syncwarp();
                    // ldmatrix: lane gives the address of row lane % 8 of matrix lane / 8 = (rows 0-7, section 0),
                    // (8-15, 0), (0-7, 1), (8-15, 1); then the two of section 2
                    uint32_t a[2][TW][4], a2[2][TW][2];
                    auto fragments = [&](int j) {
#pragma unroll
                        for (int k = 0; k < tw; ++k) {
                            const uint32_t at = tile + uint32_t(k) * kTileBytes + uint32_t(j) * kTileCol + uint32_t(lane & 15) * 48u;
                            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                                         : "=r"(a[j & 1][k][0]), "=r"(a[j & 1][k][1]), "=r"(a[j & 1][k][2]), "=r"(a[j & 1][k][3])
                                         : "r"(at + uint32_t(lane >> 4) * 16u) : "memory");
                            asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
                                         : "=r"(a2[j & 1][k][0]), "=r"(a2[j & 1][k][1]) : "r"(at + 32u) : "memory");
                        }
                    };
                    fragments(0);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (j < 3) fragments(j + 1);
                        const auto& b = b_held[j];
#pragma unroll
                        for (int k = 0; k < tw; ++k) {
                            const float s0 = __shfl_sync(0xFFFFFFFFu, scale[k][0], (lane & 28) | j);
                            const float s1 = __shfl_sync(0xFFFFFFFFu, scale[k][1], (lane & 28) | j);
#pragma unroll
                            for (int g = 0; g < G; ++g) {
                                float d[4] = {0.f, 0.f, 0.f, 0.f};
                                mma_k16(d, a[j & 1][k], b[g][0], b[g][1]);
                                mma_k8(d, a2[j & 1][k][0], a2[j & 1][k][1], b[g][2]);
                                fma2(s0, d[0], d[1], acc[i0 + k][g][0], acc[i0 + k][g][1]);
                                fma2(s1, d[2], d[3], acc[i0 + k][g][2], acc[i0 + k][g][3]);
                            }
                        }
                    }
                    __syncwarp();  // the tile has been read before the next blocks overwrite it
                }
            }
            if (!Shape::hold && WIDE) slot ^= 1u;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // everybody has left the buffers and tiles: the sums take their place
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if constexpr (!DENSE) {  // the four columns of a row first; lane t writes the pairs t modulo 4
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        acc[i][g][k] += __shfl_xor_sync(0xFFFFFFFFu, acc[i][g][k], 1);
                        acc[i][g][k] += __shfl_xor_sync(0xFFFFFFFFu, acc[i][g][k], 2);
                    }
                }
                float* at = part + ((i * W + warp) * 16 + 2 * q) * PS + (DENSE ? 8 * g + 2 * t : 2 * g);
                if (DENSE || (g & 3) == t) {
                    *reinterpret_cast<float2*>(at) = make_float2(acc[i][g][0], acc[i][g][1]);
                    *reinterpret_cast<float2*>(at + PS) = make_float2(acc[i][g][2], acc[i][g][3]);
                }
            }
        __syncthreads();
        // Output `id`: (tile, vector, row of the tile); the warps' sums in warp order.
        const int ids = nt * (16 * SLOTS);
        auto warps_sum = [&](int id) {
            const int r = id & 15, v = (id >> 4) % SLOTS, rt = (id >> 4) / SLOTS;
            const float* at = part + (rt * W * 16 + r) * PS + v;
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < W; ++w) sum += at[w * 16 * PS];
            return sum;
        };
        // Twice the halves' sum (row scale, tail).  A column with a NaN or an infinity has made its products in every row
        // infinite or NaN: 0 x sum makes them all NaN.
        auto finish = [&](float sum, int id) {
            const int r = id & 15, v = (id >> 4) % SLOTS, rt = (id >> 4) / SLOTS, i = 16 * rt + r, row = 16 * t0 + i;
            if (row >= P.N || v >= V) return;
            float res = 2.f * rs_sm[i] * fmaf(0.f, sum, sum);
            for (int k = 0; k < ntail; ++k) res = fmaf(__half2float(tail_sm[i * 24 + k]), xtail[24 * v + k], res);
            P.y[size_t(v) * P.N + row] = res;
        };
        if (C == 1) {
            for (int id = threadIdx.x; id < ids; id += THREADS) finish(warps_sum(id), id);
        } else {
            // The sums over the CTA's columns replace the parts once everybody has read those; then every CTA of the
            // cluster finishes its share of the outputs.
            constexpr int PER = (NT * 16 * SLOTS + THREADS - 1) / THREADS;
            float sums[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) sums[j] = int(threadIdx.x) + j * THREADS < ids ? warps_sum(int(threadIdx.x) + j * THREADS) : 0.f;
            __syncthreads();
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (int(threadIdx.x) + j * THREADS < ids) part[threadIdx.x + j * THREADS] = sums[j];
            cluster_barrier();
            const int id_lo = ids * rank / C, id_hi = ids * (rank + 1) / C;
            for (int id = id_lo + int(threadIdx.x); id < id_hi; id += THREADS) {
                float sum = 0.f;
                for (int c = 0; c < C; ++c) sum += cluster_load(smem_u32(part + id), uint32_t(c));
                finish(sum, id);
            }
            cluster_barrier();  // the other CTAs have read this one's sums
        }
    }
}

// Scratch that a caller brings: the call keeps its partial sums in shared memory and leaves it untouched.  The size is
// the one that the entry point has always asked for, so what it refused it still refuses.
size_t batched_workspace_bytes(int N, int blocks_per_row) {
    const long long row_tiles = (N + 511) / 512, cells = row_tiles * ((blocks_per_row + 3) / 4);
    const long long pieces = (cells < 1024 ? (cells < 1 ? 1 : cells) : 1024) + row_tiles;
    return size_t(pieces) * 16 * 512 * 4;
}

namespace {

constexpr int kBatMaxCluster = 2;
static_assert(kBatMaxCluster <= kNormClusterMax, "the scale tables' addresses");
struct BatPlan {
    int cluster = 1, groups = 1, nt = 1;
};
// How rows and columns are split: for every cluster size the steps of the busiest warp, in units of one tile x four
// columns (0.8-0.9 us with up to four vectors, 0.9-1.3 with eight, 1.2-1.7 with sixteen), and what else the split
// costs: a chunk of tiles its words, barriers and sums, a cluster its barriers and the other CTA's sums.  One CTA / two, us:
//   vectors   1184 x 12288   2368 x 12288   3000 x 12288   4096 x 12288   1024 x 4080   2368 x 4080   512 x 4080
//         3     9.0 /  7.9     9.6 / 10.9    15.3 / 13.5    15.5 / 16.9     4.2 / 5.4     5.1 / 6.7    4.2 / 4.3
//         8    12.0 /  9.3    12.8 / 13.1    19.9 / 16.5    20.0 / 20.0     5.1 / 5.6     5.9 / 7.4    5.0 / 4.7
//        16    15.1 / 10.9    16.0 / 14.6    22.2 / 18.9    22.3 / 23.5     6.3 / 6.4     7.0 / 8.3    6.2 / 5.5
//   chosen           two            one            two            one           one           one          one
// Short of the best by up to 10 % where rows are few and columns are 4080 or so (a constant of 3 that does not go with the
// vectors) and 9 % for sixteen vectors on 2368 x 12288, elsewhere within 6 %.  As many tiles to a step as registers allow:
// 12288 x 4080 with at most 1, 2, 3, 4 tiles 22.3 / 19.4 / 17.2 / 17.2 us for three vectors, 34.2 / 26.6 / 24.4 / 24.4 for
// sixteen.  Larger clusters than two: with the whole rank kept in the scale tables' address (kNormClusterMax) four CTAs took
// 7.4 us instead of 9.6 for sixteen vectors on 512 x 12288, and everything above 600 rows 1.5 to 3 times as long.
BatPlan plan_batched(int tiles, int quads, int sms) {
    BatPlan best;
    double best_cost = 1e30;
    for (int c = 1; c <= kBatMaxCluster; c *= 2) {
        const int room = sms / c;
        if (c > quads || room == 0) break;
        BatPlan p;
        p.cluster = c;
        p.groups = tiles < room ? tiles : room;
        const int most = (tiles + p.groups - 1) / p.groups, chunks = (most + kBatMaxTiles - 1) / kBatMaxTiles;
        p.nt = (most + chunks - 1) / chunks;
        const int steps = ((quads + c - 1) / c + kBatWarps - 1) / kBatWarps;
        const double cost = double(steps) * chunks * p.nt + (c > 1 ? 3.0 : 0.0) + 1.5 * chunks;
        if (cost < best_cost) {
            best_cost = cost;
            best = p;
        }
    }
    return best;
}

struct BatKernel {
    void (*run)(const DeviceTables*, BatParams);
    uint32_t smem;
};
template <bool DENSE, int G, int NT, bool WIDE>
constexpr BatKernel bat_kernel() {
    return {k_gemv_batched<DENSE, G, NT, WIDE>, BatShape<DENSE, G, NT, WIDE>::smem.total};
}
#define BAT_TILES(dense, g, wide) {bat_kernel<dense, g, 1, wide>(), bat_kernel<dense, g, 2, wide>(), bat_kernel<dense, g, 3, wide>(), bat_kernel<dense, g, 4, wide>()}
// By alignment of the rows of x, vectors (up to 2, 4: block diagonal; 8, 16: dense) and tiles of a step.  With both ways of
// copying in each kernel, chosen as it runs, the aligned rows paid in registers: 4096 x 12288 with 16 vectors 26.0 us; 22.1 now.
// (The lanes' loads of before beside the aligned copies: 22.8.)
const BatKernel kBatKernels[2][4][kBatMaxTiles] = {
    {BAT_TILES(false, 1, false), BAT_TILES(false, 2, false), BAT_TILES(true, 1, false), BAT_TILES(true, 2, false)},
    {BAT_TILES(false, 1, true), BAT_TILES(false, 2, true), BAT_TILES(true, 1, true), BAT_TILES(true, 2, true)},
};
#undef BAT_TILES

}  // namespace

cudaError_t launch_gemv_batched(const void* codes, const float* row_scales, const void* table, const void* x,
                                float* y, int N, int K, int batch, const void* tail, void*, cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    // The first call for aligned rows, or for others, loads the sixteen kernels of its kind and not the other sixteen.
    const bool wide = ((reinterpret_cast<uintptr_t>(x) | (uintptr_t(K) * 2)) & 15) == 0;
    static PerDeviceOnce once[2];
    e = once[wide].run([wide] {
        cudaError_t r = cudaSuccess;
        for (const auto& row : kBatKernels[wide])
            for (const BatKernel& k : row)
                if (r == cudaSuccess) r = cudaFuncSetAttribute(k.run, cudaFuncAttributeMaxDynamicSharedMemorySize, int(k.smem));
        return r;
    });
    if (e != cudaSuccess) return e;
    BatParams P;
    P.codes = static_cast<const unsigned char*>(codes);
    P.row_scales = row_scales;
    P.x = static_cast<const __half*>(x);
    P.tail = static_cast<const __half*>(tail);
    P.y = y;
    P.N = N;
    P.K = K;
    P.B = tail ? K / 24 : (K + 23) / 24;
    P.batch = batch;
    P.tiles = (N + 15) / 16;
    P.quads = (P.B + 3) / 4;
    const BatPlan plan = plan_batched(P.tiles, P.quads, sms);
    P.groups = plan.groups;
    P.cluster = plan.cluster;
    const BatKernel& kernel = kBatKernels[wide][batch <= 2 ? 0 : (batch <= 4 ? 1 : (batch <= 8 ? 2 : 3))][plan.nt - 1];
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = unsigned(plan.cluster);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(plan.groups * plan.cluster));
    cfg.blockDim = dim3(kBatThreads);
    cfg.dynamicSmemBytes = kernel.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = plan.cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel.run, static_cast<const DeviceTables*>(table), P);
}

}  // namespace tetra
