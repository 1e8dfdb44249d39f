// 4-bit group-quantised matrices: device layout, matrix-vector product, row dequantisation
// (Sec. 4.1 and 4.3: int4 records, groups of 128; Sec. 4.4: embedding table and output head, groups of
// 64; Sec. 5.1: dequantise with the group's scale and offset, accumulate in float32).
//
// The product is bound by HBM (4.25 or 4.5 bits per weight), so the kernel is built around bytes in
// flight and instructions per byte.  A 32-bit word of eight nibbles becomes four float16x2 operand
// registers with five logic operations:  (w & 0x000F000F) | 0x64006400 is the pair (1024 + n0, 1024 + n4),
// (w & 0x00F000F0) | 0x54005400 is (64 + n1, 64 + n5), and the same two masks on w >> 8 give n2, n6 and n3,
// n7.  The packed layout puts the nibbles where mma.sync.m16n8k16 wants them, so those registers ARE the A
// fragment of a 16-row x 16-weight tile; the activations are the B fragment (column v = vector v, so up to
// eight vectors cost the same as one), products of exact float16 values are accumulated in float32 inside
// the MMA, one accumulator per group; the biases 1024 and 64 are removed with the group's precomputed
// sum(bias_k x_k), then scale and offset are applied in float32:
//     y += scale * (D - C_group) + offset * sum_group(x).
// Tensor cores are used here as the cheapest exact multiply-accumulate (six instructions per 256 weights),
// not because the product is compute-bound: at one FFMA per weight the FP32 pipes would be the limit.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/tetra.h"
#include "../../include/tetra_q4.h"
#include "q4_common.cuh"
#include "tetra_gemv_common.cuh"

namespace tetra {
namespace {

constexpr int kQ4Threads = 512;
constexpr int kQ4CtasPerSm = 1;
constexpr int kQ4Warps = kQ4Threads / 32;

// Nibbles of two rows (v0: row g, v1: row g + 8; four consecutive columns each, column c + i at bits 4 i) as the
// packed word: columns c, c + 2, c + 1, c + 3 of row g at bits 0, 4, 16, 20, row g + 8 eight bits further up.
__device__ __forceinline__ uint32_t q4_pack_word(uint32_t v0, uint32_t v1) {
    const uint32_t even = (v0 & 0x0F0Fu) | ((v1 & 0x0F0Fu) << 16);         // columns c, c + 2 of both rows
    const uint32_t odd = ((v0 >> 4) & 0x0F0Fu) | ((v1 << 12) & 0x0F0F0000u);  // columns c + 1, c + 3
    // bytes (row g: c, c + 2; row g + 8: c, c + 2) -> nibble pairs
    const uint32_t e = (even | (even >> 4)) & 0x00FF00FFu, o = (odd | (odd >> 4)) & 0x00FF00FFu;
    return (e & 0xFFu) | ((e >> 8) & 0xFF00u) | ((o & 0xFFu) << 16) | ((o << 8) & 0xFF000000u);
}

// One warp per chunk (strip, group): lane 4 g + t reads, for every sub-tile, the 16 columns 16 t .. of rows g and
// g + 8 (eight bytes each; the four lanes of a row read one sector) and writes the lane's 16 bytes, then the row's
// scale and offset.  Bound by HBM (the matrix once in, once out); neighbouring warps take neighbouring groups, so
// the sectors of the scale tables are shared through L1.  4096 x 12288, G = 128: 10.9 us (56 MB, 5.2 TB/s);
// with a thread per packed word and byte loads 36.9 us.
template <int G>
__global__ void __launch_bounds__(256) k_q4_pack(const uint8_t* __restrict__ q, const __half* __restrict__ scale,
                                                 const __half* __restrict__ offset, unsigned char* __restrict__ packed,
                                                 int N, int K) {
    constexpr int TPG = G / 64, CH = q4_chunk_bytes(G);
    const int strips = (N + 31) / 32, groups = K / G;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // No pdl_release: the products read the packed matrix ahead of their wait (see tetra_device.cuh).
    pdl_wait();  // the matrix may come from, the packed one be read by, the kernel before
    const size_t chunks = size_t(strips) * groups;
    for (size_t chunk = (blockIdx.x * size_t(blockDim.x) + threadIdx.x) >> 5; chunk < chunks;
         chunk += (size_t(gridDim.x) * blockDim.x) >> 5) {
        const int strip = int(chunk / groups), group = int(chunk - size_t(strip) * groups);
        uint2 v[TPG][2][2];  // [tile][sub-tile][row g, row g + 8]
#pragma unroll
        for (int j = 0; j < TPG; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const int row = 32 * strip + 16 * h + g + 8 * half;
                    const uint2* src = reinterpret_cast<const uint2*>(q + size_t(row) * (K / 2) + group * (G / 2) + 32 * j + 8 * t);
                    v[j][h][half] = row < N ? __ldg(src) : make_uint2(0u, 0u);
                }
        const int row = 32 * strip + lane;
        uint32_t so = 0;
        if (row < N) {
            const size_t at = size_t(row) * groups + group;
            so = uint32_t(__half_as_ushort(__ldg(scale + at))) | (uint32_t(__half_as_ushort(__ldg(offset + at))) << 16);
        }
        unsigned char* dst = packed + chunk * CH;
#pragma unroll
        for (int j = 0; j < TPG; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint2 a = v[j][h][0], b = v[j][h][1];
                *reinterpret_cast<uint4*>(dst + j * 1024 + h * 512 + lane * 16) =
                    make_uint4(q4_pack_word(a.x & 0xFFFFu, b.x & 0xFFFFu), q4_pack_word(a.x >> 16, b.x >> 16),
                               q4_pack_word(a.y & 0xFFFFu, b.y & 0xFFFFu), q4_pack_word(a.y >> 16, b.y >> 16));
            }
        *reinterpret_cast<uint32_t*>(dst + TPG * 1024 + lane * 4) = so;
    }
}

// A CTA owns a contiguous range of 32-row strips (equal shares), and its 16 warps cut the CTA's chunks, in
// memory order, into 16 equal contiguous ranges: every warp streams one contiguous piece of the matrix
// through a ring of DEPTH slots in shared memory (cp.async, DEPTH - 1 chunks ahead).  Per chunk: the
// accumulators of the two 16-row sub-tiles start at minus the group's sum(bias_k x_k), every 64-column tile
// adds four MMAs per sub-tile (the activations' B fragments are shared by both), then
//     acc += scale * D + offset * sum_group(x).
// A strip that lies wholly inside a warp's range is stored directly; a strip cut by a range boundary leaves
// one piece per warp in shared memory, and after one CTA barrier the pieces are added in warp order; which strips those
// are is worked out while the kernel waits for its predecessor (looked for afterwards, piece by piece, it was 2.2 us of
// a 5.1 us launch: 1024 x 4096, G = 128, now 3.7 us).
// Addresses advance by running pointers: the loop body is dequantise, multiply, scale.
// XS: the activations are staged in shared memory (rows padded by 16 bytes so that the eight vectors' reads
// fall into different banks); otherwise they are read through L1.
template <int G, int DEPTH, bool XS>
__global__ void __launch_bounds__(kQ4Threads, kQ4CtasPerSm)
k_q4_gemv(const unsigned char* __restrict__ packed, const __half* __restrict__ x, float* __restrict__ y, int N, int K,
          int batch) {
    constexpr int TPG = G / 64, CH = q4_chunk_bytes(G), PIECES = CH / 16;
    extern __shared__ __align__(16) unsigned char q4_smem[];
    const int groups = K / G, strips = (N + 31) / 32;
    float2* gs = reinterpret_cast<float2*>(q4_smem);                        // [groups][8]: (sum x, -sum bias x)
    float* pieces = reinterpret_cast<float*>(q4_smem + size_t(groups) * 64);  // [warps][2][256]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int kPieceBytes = kQ4Warps * 2 * 1024;
    const uint32_t ring = smem_u32(q4_smem + size_t(groups) * 64 + kPieceBytes) + uint32_t(warp) * (DEPTH * CH);
    unsigned char* xs_base = q4_smem + size_t(groups) * 64 + kPieceBytes + size_t(kQ4Warps) * DEPTH * CH;
    const uint32_t xs_stride = uint32_t(K) * 2u + 16u;  // bytes per staged vector
    const int g = lane >> 2, t = lane & 3;
    pdl_release();

    // this CTA's strips, this warp's chunks (local index n = local strip * groups + group)
    const int strip_begin = int(size_t(blockIdx.x) * strips / gridDim.x);
    const int strip_end = int((size_t(blockIdx.x) + 1) * strips / gridDim.x);
    const uint32_t cta_chunks = uint32_t(strip_end - strip_begin) * uint32_t(groups);
    // every range non-empty: fewer chunks than warps leave warps over
    const uint32_t ranges = min(cta_chunks, uint32_t(kQ4Warps));
    auto range_begin = [&](uint32_t w) { return cta_chunks <= uint32_t(kQ4Warps) ? min(w, cta_chunks) : uint32_t(uint64_t(w) * cta_chunks / kQ4Warps); };
    const uint32_t n_begin = range_begin(uint32_t(warp)), n_end = range_begin(uint32_t(warp) + 1);
    // running addresses: f_src = next chunk to copy (this lane's 16 bytes of each 512), f_todo = chunks left to
    // copy; slot_lane = this lane's 16 bytes in the slot being consumed; the slot consumed last is refilled
    const unsigned char* f_src = packed + (size_t(strip_begin) * groups + n_begin) * CH + lane * 16;
    int f_todo = int(n_end - n_begin);
    const uint32_t ring_lane = ring + lane * 16, ring_lane_end = ring_lane + DEPTH * CH;
    const bool tail_lane = lane < PIECES % 32;  // lanes that copy the last, partial group of 16-byte pieces
    auto fetch_into = [&](uint32_t dst_lane) {
        if (f_todo > 0) {
#pragma unroll
            for (int i = 0; i < PIECES / 32; ++i) q4_cp_async16(dst_lane + i * 512, f_src + i * 512);
            if (PIECES % 32 != 0 && tail_lane) q4_cp_async16(dst_lane + (PIECES / 32) * 512, f_src + (PIECES / 32) * 512);
            f_src += CH;
        }
        --f_todo;
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per call, empty or not
    };
#pragma unroll
    for (int i = 0; i < DEPTH - 1; ++i) fetch_into(ring_lane + i * CH);  // the weights do not depend on the preceding kernel

    // cut[w]: the strip that begins in warp w's range and goes on beyond it, and over how many ranges it stretches in all
    // (0: there is none); known from here on, needed at the end
    __shared__ int2 cut[kQ4Warps];
    if (threadIdx.x < kQ4Warps) {
        const uint32_t w = threadIdx.x, begin = range_begin(w), end = range_begin(w + 1);
        int2 c = make_int2(0, 0);
        if (begin < end) {
            const uint32_t s = (end - 1) / uint32_t(groups), s_begin = s * uint32_t(groups), s_end = s_begin + uint32_t(groups);
            if (s_begin >= begin && s_end > end) {
                uint32_t k = w + 1;
                while (k < ranges && range_begin(k) < s_end) ++k;
                c = make_int2(int(s), int(k - w));
            }
        }
        cut[w] = c;
    }
    pdl_wait();  // x may come from the preceding kernel
    // The activations, eight to a thread (into shared memory if they fit), and on the way, per (group, vector), the sum of
    // x and minus the sum of bias_k x_k, bias 1024 for k % 4 in {0, 1}, 64 for {2, 3}: G / 8 neighbouring lanes combined
    // by shuffles in a fixed order.
    {
        const uint32_t per_vec = uint32_t(K) / 8u, total = per_vec * uint32_t(batch), inv = 0xFFFFFFFFu / per_vec + 1u;
        constexpr int AHEAD = 4;  // loads in flight per thread
        for (uint32_t i0 = warp * 32; i0 < total; i0 += AHEAD * kQ4Threads) {  // whole warps, for the shuffles
            uint4 u[AHEAD];
#pragma unroll
            for (int j = 0; j < AHEAD; ++j) {
                const uint32_t i = i0 + uint32_t(j * kQ4Threads + lane), v = __umulhi(i, inv);
                u[j] = i < total ? __ldg(reinterpret_cast<const uint4*>(x + size_t(v) * K) + (i - v * per_vec)) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int j = 0; j < AHEAD; ++j) {
                if (i0 + uint32_t(j * kQ4Threads) >= total) break;  // warp-uniform
                const uint32_t i = i0 + uint32_t(j * kQ4Threads + lane), v = __umulhi(i, inv), c8 = i - v * per_vec;
                if (XS && i < total) *reinterpret_cast<uint4*>(xs_base + size_t(v) * xs_stride + size_t(c8) * 16) = u[j];
                const float2 a0 = __half22float2(*reinterpret_cast<const __half2*>(&u[j].x)), b0 = __half22float2(*reinterpret_cast<const __half2*>(&u[j].y));
                const float2 a1 = __half22float2(*reinterpret_cast<const __half2*>(&u[j].z)), b1 = __half22float2(*reinterpret_cast<const __half2*>(&u[j].w));
                float lo = (a0.x + a0.y) + (a1.x + a1.y), hi = (b0.x + b0.y) + (b1.x + b1.y);  // k % 4 in {0, 1} / {2, 3}
#pragma unroll
                for (int o = G / 16; o >= 1; o >>= 1) {
                    lo += __shfl_xor_sync(0xFFFFFFFFu, lo, o);
                    hi += __shfl_xor_sync(0xFFFFFFFFu, hi, o);
                }
                if (lane % (G / 8) == 0 && i < total) gs[c8 / (G / 8) * 8 + v] = make_float2(lo + hi, -(1024.f * lo + 64.f * hi));
            }
        }
    }
    for (int i = threadIdx.x; i < groups * 8; i += kQ4Threads)
        if ((i & 7) >= batch) gs[i] = make_float2(0.f, 0.f);
    if (XS && threadIdx.x < kQ4TileZeros / 16) reinterpret_cast<uint4*>(xs_base + size_t(batch) * xs_stride)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();

    // Column g of B is vector g.  Columns at or beyond batch are never stored and read zeros wherever the walk is
    // (x_step 0): multiplying zeros takes less power, and large matrices run at the board's limit.
    const bool fed = g < batch;
    const uint32_t x_step = fed ? 2u * G : 0u;
    // this lane's 16 activations of the first tile of group 0: a shared address or a pointer
    const auto x_lane = [&] {
        if constexpr (XS) return smem_u32(xs_base) + (fed ? uint32_t(g) * xs_stride + 32u * t : uint32_t(batch) * xs_stride);
        else return fed ? reinterpret_cast<const unsigned char*>(x + size_t(g) * K + 16 * t) : reinterpret_cast<const unsigned char*>(q4_zeros);
    }();
    const uint32_t gs_lane = smem_u32(gs) + uint32_t(t) * 16;
    uint32_t slot_lane = ring_lane;                       // slot being consumed
    uint32_t refill_lane = ring_lane + (DEPTH - 1) * CH;  // slot consumed last (empty at the start)
    const uint32_t so_delta = uint32_t(TPG * 1024 + g * 4) - uint32_t(lane * 16);  // slot_lane -> this lane's scale records
    int gi = int(n_begin % uint32_t(groups));
    int strip = strip_begin + int(n_begin / uint32_t(groups));
    uint32_t left = n_end - n_begin;
    while (left > 0) {
        // one segment: the chunks of this warp that belong to one strip
        const int seg_first = gi;
        const uint32_t seg_len = min(uint32_t(groups - gi), left);
        auto xo = x_lane + uint32_t(gi) * x_step;
        uint32_t gsp = gs_lane + uint32_t(gi) * 64;
        float acc[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[h][i] = 0.f;
        for (uint32_t c = 0; c < seg_len; ++c) {
            uint32_t cs[4];  // (sum x, -sum bias x) of vectors 2 t, 2 t + 1
            q4_lds128(gsp, cs);
            [[maybe_unused]] uint32_t xl[TPG][8];
            if constexpr (!XS) load_group<TPG>(xo, xl);  // ahead of the copies: see there
            fetch_into(refill_lane);
            q4_cp_async_wait<DEPTH - 1>();  // this chunk has landed
            __syncwarp();
            float d[2][4];
#pragma unroll
            for (int j = 0; j < TPG; ++j) {
                uint32_t xr[8];
                if constexpr (XS) {
                    uint32_t lo[4], hi[4];
                    q4_lds128(xo + 128 * j, lo);
                    q4_lds128(xo + 128 * j + 16, hi);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        xr[i] = lo[i];
                        xr[4 + i] = hi[i];
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) xr[i] = xl[j][i];
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t ww[4];
                    q4_lds128(slot_lane + j * 1024 + h * 512, ww);
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        uint32_t a[4];
                        const uint32_t w8 = ww[m] >> 8;
                        a[0] = lop_and_or(ww[m], 0x000F000Fu, 0x64006400u);  // row g,     columns c, c+1   (1024 + n)
                        a[1] = lop_and_or(w8, 0x000F000Fu, 0x64006400u);     // row g + 8, columns c, c+1
                        a[2] = lop_and_or(ww[m], 0x00F000F0u, 0x54005400u);  // row g,     columns c+2, c+3 (64 + n)
                        a[3] = lop_and_or(w8, 0x00F000F0u, 0x54005400u);     // row g + 8, columns c+2, c+3
                        if (j == 0 && m == 0)
                            mma_f16_first(d[h], a, xr[0], xr[1], __uint_as_float(cs[1]), __uint_as_float(cs[3]));
                        else
                            mma_f16(d[h], a, xr[2 * m], xr[2 * m + 1]);
                    }
                }
            }
            // this lane's results: rows 16 h + g (i = 0, 1) and 16 h + g + 8 (i = 2, 3), vectors 2 t + (i & 1)
            const float sx_even = __uint_as_float(cs[0]), sx_odd = __uint_as_float(cs[2]);
            const uint32_t so_lane = slot_lane + so_delta;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t so0 = lds32(so_lane + 64 * h);
                const uint32_t so1 = lds32(so_lane + 64 * h + 32);
                const float2 r0 = __half22float2(*reinterpret_cast<const __half2*>(&so0));  // (scale, offset)
                const float2 r1 = __half22float2(*reinterpret_cast<const __half2*>(&so1));
                fma2(r0.y, sx_even, sx_odd, acc[h][0], acc[h][1]);  // offset * sum(x), vectors 2 t and 2 t + 1
                fma2(r0.x, d[h][0], d[h][1], acc[h][0], acc[h][1]);  // scale * (sum q x)
                fma2(r1.y, sx_even, sx_odd, acc[h][2], acc[h][3]);
                fma2(r1.x, d[h][2], d[h][3], acc[h][2], acc[h][3]);
            }
            __syncwarp();  // every lane has read the slot before the next refill targets it
            refill_lane = slot_lane;
            slot_lane += CH;
            if (slot_lane == ring_lane_end) slot_lane = ring_lane;
            xo += x_step;
            gsp += 64;
        }
        left -= seg_len;
        gi += int(seg_len);
        // element e = 8 lane + 4 h + i is (row 16 h + g + 8 (i / 2), vector 2 t + (i % 2)) of the strip
        if (seg_first == 0 && gi == groups) {  // the whole strip was this warp's
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = 32 * strip + 16 * h + g + 8 * (i >> 1), v = 2 * t + (i & 1);
                    if (row < N && v < batch) y[size_t(v) * N + row] = acc[h][i];
                }
        } else {  // a strip shared with a neighbouring warp: leave a piece (slot 0: it began before this range, 1: it ends beyond)
            float* mine = pieces + (2 * warp + (seg_first != 0 ? 0 : 1)) * 256 + 8 * lane;
            *reinterpret_cast<float4*>(mine) = make_float4(acc[0][0], acc[0][1], acc[0][2], acc[0][3]);
            *reinterpret_cast<float4*>(mine + 4) = make_float4(acc[1][0], acc[1][1], acc[1][2], acc[1][3]);
        }
        if (gi == groups) {
            gi = 0;
            ++strip;
        }
    }
    q4_cp_async_wait<0>();
    __syncthreads();
    // The strips that a range boundary cuts: warp w's second piece, then the first pieces of the warps after it.  Half
    // of the CTA's threads takes the even w, half the odd ones; a thread is one of the 256 results of a strip.
    const int e = threadIdx.x & 255, el = e >> 3, h = (e >> 2) & 1, i = e & 3;
    const int r_in = 16 * h + (el >> 2) + 8 * (i >> 1), v = 2 * (el & 3) + (i & 1);
#pragma unroll 1
    for (int w = int(threadIdx.x >> 8); w < kQ4Warps; w += kQ4Threads / 256) {
        const int2 c = cut[w];
        if (c.y == 0) continue;
        const float* at = pieces + 2 * w * 256 + e;
        float total = at[256];
#pragma unroll
        for (int k0 = 1; k0 < kQ4Warps; k0 += 5) {  // five loads at a time
            if (k0 >= c.y) break;
            float p[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) p[k] = k0 + k < c.y ? at[(k0 + k) * 512] : 0.f;
#pragma unroll
            for (int k = 0; k < 5; ++k) total += p[k];
        }
        const int row = 32 * (strip_begin + c.x) + r_in;
        if (row < N && v < batch) y[size_t(v) * N + row] = total;
    }
}

// Float16 weights of the rows of some tokens (Sec. 4.4).  A thread takes the 16 columns 16 t .. of one 64-column
// tile: one 16-byte load (a quarter of the 64 bytes in which the tile holds the row and its neighbour eight rows
// away), the row's scale record, 32 bytes out.  WIDE: `out` allows 16-byte stores.  A short call is the chain token
// number -> weights -> store, and only resident warps hide it: one token per CTA row (two or four tokens a thread,
// their loads together, take 5.8 and 8.4 us where one takes 4.8).
// 1024 tokens x 4096: 4.8 us; with a thread per four columns 7.9 us.
template <int G, bool WIDE>
__global__ void __launch_bounds__(256) k_q4_rows(const unsigned char* __restrict__ packed, const int32_t* __restrict__ ids,
                                                 int count, __half* __restrict__ out, int N, int K) {
    constexpr int CH = q4_chunk_bytes(G);
    const int groups = K / G, per_row = K / 16;  // threads per token
    pdl_release();
    const int at = blockIdx.x * blockDim.x + threadIdx.x;  // tile quarter of the row
    if (at >= per_row) return;
    const int c = 16 * at, group = c / G, j = (c % G) >> 6, t = at & 3;
    pdl_wait();  // the ids may come from the preceding kernel
    for (int tok = blockIdx.y; tok < count; tok += gridDim.y) {
        const int row = __ldg(ids + tok);
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        uint32_t rec = 0u;
        if (row >= 0 && row < N) {  // otherwise the record stays zero, and with it the row
            const int strip = row >> 5, rr = row & 31, h = rr >> 4, g = rr & 7;
            const unsigned char* chunk = packed + (size_t(strip) * groups + group) * CH;
            w = __ldg(reinterpret_cast<const uint4*>(chunk + j * 1024 + h * 512 + (g * 4 + t) * 16));
            rec = __ldg(reinterpret_cast<const uint32_t*>(chunk + (G / 64) * 1024 + rr * 4));
        }
        const int half = (row >> 3) & 1;
        const float2 sc = __half22float2(*reinterpret_cast<const __half2*>(&rec));
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
        uint32_t r[8];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t v = ww[m] >> (8 * half);
            const float n0 = float(v & 15u), n1 = float((v >> 16) & 15u);        // columns 4 m, 4 m + 1
            const float n2 = float((v >> 4) & 15u), n3 = float((v >> 20) & 15u);  // columns 4 m + 2, 4 m + 3
            const __half2 lo = __floats2half2_rn(__fmaf_rn(sc.x, n0, sc.y), __fmaf_rn(sc.x, n1, sc.y));
            const __half2 hi = __floats2half2_rn(__fmaf_rn(sc.x, n2, sc.y), __fmaf_rn(sc.x, n3, sc.y));
            r[2 * m] = *reinterpret_cast<const uint32_t*>(&lo);
            r[2 * m + 1] = *reinterpret_cast<const uint32_t*>(&hi);
        }
        __half* dst = out + size_t(tok) * K + c;
        if (WIDE) {
            reinterpret_cast<uint4*>(dst)[0] = make_uint4(r[0], r[1], r[2], r[3]);
            reinterpret_cast<uint4*>(dst)[1] = make_uint4(r[4], r[5], r[6], r[7]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) reinterpret_cast<uint2*>(dst)[k] = make_uint2(r[2 * k], r[2 * k + 1]);
        }
    }
}

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }
inline int cuda_status(cudaError_t e) { return e == cudaSuccess ? TETRA_OK : TETRA_ERR_CUDA; }

int check_shape(int N, int K, int G) {
    if (N <= 0 || K <= 0 || K > TETRA_Q4_MAX_K) return TETRA_ERR_SHAPE;
    if ((G != 64 && G != 128) || K % G) return TETRA_ERR_SHAPE;
    return TETRA_OK;
}

constexpr size_t kQ4SmemLimit = 224 * 1024 / kQ4CtasPerSm - 2048;

template <int G, int DEPTH>
constexpr size_t q4_smem_bytes(int K, int batch, bool staged) {
    return size_t(K / G) * 64 + size_t(kQ4Warps) * 2048 + size_t(kQ4Warps) * DEPTH * q4_chunk_bytes(G) +
           (staged ? size_t(batch) * (size_t(K) * 2 + 16) + kQ4TileZeros : 0);
}

template <int G, int DEPTH, bool XS>
cudaError_t launch_q4_variant(const void* packed, const void* x, float* y, int N, int K, int batch, int sms,
                              cudaStream_t s) {
    const int strips = (N + 31) / 32;
    const int grid = strips < kQ4CtasPerSm * sms ? strips : kQ4CtasPerSm * sms;
    const size_t smem = q4_smem_bytes<G, DEPTH>(K, batch, XS);
    static PerDeviceOnce once;  // per instantiation
    cudaError_t e = once.run([] {
        return cudaFuncSetAttribute(k_q4_gemv<G, DEPTH, XS>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kQ4SmemLimit));
    });
    if (e != cudaSuccess) return e;
    if (smem > kQ4SmemLimit) return cudaErrorInvalidValue;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(kQ4Threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_q4_gemv<G, DEPTH, XS>, static_cast<const unsigned char*>(packed),
                              static_cast<const __half*>(x), y, N, K, batch);
}

template <int G, int DEPTH>
cudaError_t launch_q4_gemv(const void* packed, const void* x, float* y, int N, int K, int batch, int sms,
                           cudaStream_t s) {
    // Staged wherever they fit: read through L1 the activations queue behind the weights' copies, which the same unit
    // takes in order (see q4_list.cu).
    if (q4_smem_bytes<G, DEPTH>(K, batch, true) <= kQ4SmemLimit)
        return launch_q4_variant<G, DEPTH, true>(packed, x, y, N, K, batch, sms, s);
    return launch_q4_variant<G, DEPTH, false>(packed, x, y, N, K, batch, sms, s);
}

}  // namespace
}  // namespace tetra

using namespace tetra;

extern "C" {

size_t tetra_q4_packed_bytes(int N, int K, int G) {
    if (check_shape(N, K, G) != TETRA_OK) return 0;
    return size_t((N + 31) / 32) * (K / G) * q4_chunk_bytes(G);
}

int tetra_q4_pack(const void* q_dev, const void* scale_dev, const void* offset_dev, void* packed_dev,
                  size_t packed_bytes, int N, int K, int G, void* stream) {
    if (!q_dev || !scale_dev || !offset_dev || !packed_dev) return TETRA_ERR_NULL;
    const int rc = check_shape(N, K, G);
    if (rc != TETRA_OK) return rc;
    if (!aligned(q_dev, 16) || !aligned(scale_dev, 16) || !aligned(offset_dev, 16) || !aligned(packed_dev, 16))
        return TETRA_ERR_ALIGN;
    const size_t need = tetra_q4_packed_bytes(N, K, G);
    if (packed_bytes < need) return TETRA_ERR_SIZE;
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return TETRA_ERR_CUDA;
    const size_t chunks = size_t((N + 31) / 32) * (K / G);
    const size_t ctas = (chunks + 7) / 8, most = size_t(sms) * 64;  // a warp per chunk
    const unsigned grid = unsigned(ctas < most ? ctas : most);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const auto* q = static_cast<const uint8_t*>(q_dev);
    const auto *scale = static_cast<const __half*>(scale_dev), *offset = static_cast<const __half*>(offset_dev);
    auto* packed = static_cast<unsigned char*>(packed_dev);
    return cuda_status(launch_pdl(G == 128 ? k_q4_pack<128> : k_q4_pack<64>, int(grid), 256, 0, s, q, scale, offset, packed, N, K));
}

int tetra_q4_gemv(const void* packed_dev, const void* x_dev, float* y_dev, int N, int K, int G, int batch,
                  void* stream) {
    if (!packed_dev || !x_dev || !y_dev) return TETRA_ERR_NULL;
    const int rc = check_shape(N, K, G);
    if (rc != TETRA_OK) return rc;
    if (batch < 1 || batch > TETRA_Q4_MAX_BATCH) return TETRA_ERR_BATCH;
    if (!aligned(packed_dev, 16) || !aligned(x_dev, 16) || !aligned(y_dev, 4)) return TETRA_ERR_ALIGN;
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return TETRA_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return cuda_status(G == 128 ? launch_q4_gemv<128, 3>(packed_dev, x_dev, y_dev, N, K, batch, sms, s)
                                : launch_q4_gemv<64, 6>(packed_dev, x_dev, y_dev, N, K, batch, sms, s));
}

int tetra_q4_rows(const void* packed_dev, const int32_t* ids_dev, int count, void* out_dev, int N, int K, int G,
                  void* stream) {
    if (count == 0) return TETRA_OK;
    if (!packed_dev || !ids_dev || !out_dev) return TETRA_ERR_NULL;
    const int rc = check_shape(N, K, G);
    if (rc != TETRA_OK) return rc;
    if (count < 0) return TETRA_ERR_SHAPE;
    if (!aligned(packed_dev, 16) || !aligned(ids_dev, 4) || !aligned(out_dev, 8)) return TETRA_ERR_ALIGN;
    // a thread per 16 columns, a CTA row per token
    const int threads = K / 16 < 256 ? K / 16 : 256, gx = (K / 16 + threads - 1) / threads;
    const int gy = count < 65535 ? count : 65535;
    const bool wide = aligned(out_dev, 16);
    auto launch = [&](auto kernel) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(unsigned(gx), unsigned(gy));
        cfg.blockDim = dim3(unsigned(threads));
        cfg.stream = static_cast<cudaStream_t>(stream);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cuda_status(cudaLaunchKernelEx(&cfg, kernel, static_cast<const unsigned char*>(packed_dev), ids_dev, count,
                                              static_cast<__half*>(out_dev), N, K));
    };
    if (G == 128) return wide ? launch(k_q4_rows<128, true>) : launch(k_q4_rows<128, false>);
    return wide ? launch(k_q4_rows<64, true>) : launch(k_q4_rows<64, false>);
}

}  // extern "C"
