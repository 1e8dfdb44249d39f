// Decode-only kernels and the HBM code layout (pack) kernel.
#include "tetra_gemv_common.cuh"

namespace tetra {

// ---------------------------------------------------------------------------
// tetra_decode_blocks: file-order words -> 24 coordinates (+ m, g).  One thread
// per block; the paper-format tables are read through the read-only cache.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_decode_file(const uint8_t* __restrict__ codes,
                                                     const DeviceTables* __restrict__ tab,
                                                     int8_t* __restrict__ y_out, uint8_t* __restrict__ mg_out,
                                                     size_t nblocks) {
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < nblocks;
         i += size_t(gridDim.x) * blockDim.x) {
        int y[24], m, g;
        decode_file_word(&tab->paper, load_file_word(codes, i), y, &m, &g);
        uint32_t* dst = reinterpret_cast<uint32_t*>(y_out + 24 * i);  // 24 i is a multiple of 4
#pragma unroll
        for (int k = 0; k < 6; ++k)
            dst[k] = uint32_t(y[4 * k] & 0xFF) | (uint32_t(y[4 * k + 1] & 0xFF) << 8) |
                     (uint32_t(y[4 * k + 2] & 0xFF) << 16) | (uint32_t(y[4 * k + 3] & 0xFF) << 24);
        if (mg_out) {
            mg_out[2 * i] = uint8_t(m);
            mg_out[2 * i + 1] = uint8_t(g);
        }
    }
}

// ---------------------------------------------------------------------------
// Packed layout.  Rows are taken in groups of eight; for row group G and block
// column c the eight words form a 48-byte record split into three 16-byte
// parts, stored as  packed[(G * 3 + part) * B + c]  (uint4 units):
//   part 0: w0 of rows 8G+0..3      part 1: w0 of rows 8G+4..7
//   part 2: w1 of rows 8G+0..7 (two per 32-bit lane, even row in the low half)
// so a warp whose lanes own consecutive columns reads 512 contiguous bytes per
// part.  Rows beyond N are the all-zero word (the origin).
//
// A lane per record (row group, column).  Bound by HBM (six bytes in, six out per word) once the trellis map, one
// random lookup per word, is in shared memory and a word is one 4-byte and one 2-byte load, all 16 loads of a record
// in flight.  12288 x 4096 (25 MB), one packing behind another: 8.1 us, 3.1 TB/s (7.6 us if each one released the next
// while it runs, which packing may not: see tetra_device.cuh).  With the map and a row permutation read through L1 and
// three 2-byte loads a packing took 3 us more.
// ---------------------------------------------------------------------------
// The (row group, 32 columns) items of a warp, every `warps`-th of them in row-major order, without a division per item.
struct ItemWalk {
    int G, cg, step_G, step_cg, col_groups;
    __device__ __forceinline__ ItemWalk(int warp, int warps, int col_groups_) : col_groups(col_groups_) {
        G = warp / col_groups;
        cg = warp - G * col_groups;
        step_G = warps / col_groups;
        step_cg = warps - step_G * col_groups;
    }
    __device__ __forceinline__ void next() {
        G += step_G;
        cg += step_cg;
        if (cg >= col_groups) {
            cg -= col_groups;
            ++G;
        }
    }
};

__global__ void __launch_bounds__(256, 4) k_pack(const uint8_t* __restrict__ codes,
                                                 const DeviceTables* __restrict__ tab,
                                                 uint4* __restrict__ packed, int N, int B) {
    __shared__ uint16_t abx[4096];
    // No pdl_release: the products read codes ahead of their wait (see tetra_device.cuh).
    for (int i = threadIdx.x; i < 512; i += blockDim.x)
        reinterpret_cast<uint4*>(abx)[i] = __ldg(reinterpret_cast<const uint4*>(tab->trellis_to_abx) + i);
    __syncthreads();
    pdl_wait();  // the words may come from, the packed matrix be read by, the kernel before
    const int groups = (N + 7) / 8, lane = threadIdx.x & 31;
    const uint32_t row_bytes = uint32_t(B) * 6u;
    for (ItemWalk it((blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5, (B + 31) / 32); it.G < groups; it.next()) {
        const int G = it.G, c = min(it.cg * 32 + lane, B - 1), rows = min(8, N - 8 * G);
        // a word is 2-byte aligned: its 4-byte aligned part (first or last four bytes) and the other two bytes
        const uint8_t* first = codes + (size_t(8 * G) * B + c) * 6;
        uint32_t four[8], two[8], back[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint8_t* at = first + uint32_t(min(r, rows - 1)) * row_bytes;
            back[r] = uint32_t(reinterpret_cast<uintptr_t>(at)) & 2u;
            four[r] = __ldg(reinterpret_cast<const uint32_t*>(at + back[r]));
            two[r] = __ldg(reinterpret_cast<const unsigned short*>(at + 4 - 2 * back[r]));
        }
        uint32_t w0[8], w1[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint64_t w = back[r] ? uint64_t(two[r]) | (uint64_t(four[r]) << 16) : uint64_t(four[r]) | (uint64_t(two[r]) << 32);
            file_to_device_word(w, abx[trellis_path(w)], &w0[r], &w1[r]);
            if (r >= rows) w0[r] = w1[r] = 0u;  // padding rows: the all-zero device word
        }
        if (it.cg * 32 + lane >= B) continue;
        uint4* rec = packed + size_t(G) * 3 * B + c;
        rec[0] = make_uint4(w0[0], w0[1], w0[2], w0[3]);
        rec[B] = make_uint4(w0[4], w0[5], w0[6], w0[7]);
        rec[2 * size_t(B)] = make_uint4(w1[0] | (w1[1] << 16), w1[2] | (w1[3] << 16),
                                        w1[4] | (w1[5] << 16), w1[6] | (w1[7] << 16));
    }
}

// ---------------------------------------------------------------------------
// tetra_decode_packed: the GEMV's own decoder, emitting coordinates instead of
// multiplying.  A warp per (row group, 32 columns), the next item's record on its way meanwhile; a row's 768 bytes go
// through shared memory, so that they leave as contiguous 16-byte stores (a lane's 24 bytes, stored word by word,
// touch every sector six times).  12288 x 4096 (67 MB, 10.2 us at the copy bandwidth): 14.5 us a call one behind another.
// Captured alone (19.0 us): 136 warp-instructions per 32 blocks; while warps are active, 76 % of the launch, the L1 and
// shared-memory pipe is 75 % busy (table lookups, rows staged and read back) and issue slots 56 %; warps wait for
// their first records (long scoreboard 3.0 of 12 stall cycles per instruction: two items a warp) and for the logic
// pipe (1.8).  Direct stores made it 17 us longer.
// ---------------------------------------------------------------------------
constexpr int kEmitThreads = 256;
constexpr int kEmitStage = 2 * 768;  // two rows of 32 blocks at a time

// Coordinates of a block in file order, four int8 per word.  With a nibble's sign bit flipped it is z + 8, so
// y = -(2 z + p) = (16 - p) - 2 (z + 8), bytewise with 128 added so that no byte borrows.
__device__ __forceinline__ void file_order(const NibbleBlock& nb, uint32_t (&out)[6]) {
    const uint32_t top = 0x90909090u - ((nb.p4 >> 2) & 1u) * 0x01010101u;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const uint32_t z = nb.z[s];
        const uint32_t hi = (top - (((z >> 3) & 0x1E1E1E1Eu) ^ 0x10101010u)) ^ 0x80808080u;  // coordinates 2, 6, 3, 7
        const uint32_t lo = (top - (((z << 1) & 0x1E1E1E1Eu) ^ 0x10101010u)) ^ 0x80808080u;  // coordinates 0, 4, 1, 5
        static_assert(word_coordinate(0, 1) == 6 && word_coordinate(1, 2) == 1, "order of the nibbles");
        out[2 * s] = prmt(lo, hi, 0x6420u);
        out[2 * s + 1] = prmt(lo, hi, 0x7531u);
    }
}

// WIDTH: alignment of a row of y in bytes that the stores may use, 16, 8 or 4 (4: mg goes out bytewise).
template <int WIDTH>
__global__ void __launch_bounds__(kEmitThreads, 4)
k_decode_packed(const uint4* __restrict__ packed, const DeviceTables* __restrict__ tab, int8_t* __restrict__ y_out,
                uint8_t* __restrict__ mg_out, int N, int B) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_release();
    unsigned char* base = stage_fast_tables(tab, smem);
    const uint32_t sm_tab = smem_u32(base);
    __syncthreads();
    pdl_wait();  // the packed matrix may come from, the outputs be read by, the kernel before
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* stage = base + kFastBytes + warp * kEmitStage;
    const int groups = (N + 7) / 8;
    uint4 lo, hi, w1;
    auto load = [&](const ItemWalk& at) {
        const uint4* rec = packed + size_t(at.G) * 3 * B + min(at.cg * 32 + lane, B - 1);
        lo = __ldg(rec);
        hi = __ldg(rec + B);
        w1 = __ldg(rec + 2 * size_t(B));
    };
    // a lane's units of the copy out: unit `lane + 32 k` of two rows
    constexpr int kUnits = 768 / WIDTH, kTurns = 2 * kUnits / 32;
    uint32_t unit_at[kTurns], unit_off[kTurns];
    const uint32_t row_bytes = uint32_t(B) * 24u;
#pragma unroll
    for (int k = 0; k < kTurns; ++k) {
        const int u = lane + 32 * k, r = u >= kUnits ? 1 : 0;
        unit_at[k] = uint32_t(u - r * kUnits) * WIDTH;       // inside its row
        unit_off[k] = unit_at[k] + (r ? row_bytes : 0u);
    }
    ItemWalk it((blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5, (B + 31) / 32);
    if (it.G < groups) load(it);
    while (it.G < groups) {
        const int G = it.G, c0 = it.cg * 32, cols = min(32, B - c0), rows = min(8, N - 8 * G);
        const uint32_t w0[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        const uint32_t w1p[4] = {w1.x, w1.y, w1.z, w1.w};
        it.next();
        if (it.G < groups) load(it);
        const size_t block0 = size_t(8 * G) * B + c0;
        int8_t* y_pair = y_out + block0 * 24;
        const bool mg_lane = mg_out && lane < cols;
        uint8_t* mg_at = mg_out + 2 * (block0 + lane);
#pragma unroll
        for (int r0 = 0; r0 < 8; r0 += 2) {
            __syncwarp();  // the staged rows of the turn before have been read
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                NibbleBlock nb;
                if (r) decode_nibbles<true>(sm_tab, w0[r0 + 1], w1p[r0 >> 1], nb);
                else decode_nibbles<false>(sm_tab, w0[r0], w1p[r0 >> 1], nb);
                uint32_t y[6];
                file_order(nb, y);
                uint2* dst = reinterpret_cast<uint2*>(stage + r * 768 + lane * 24);
#pragma unroll
                for (int k = 0; k < 3; ++k) dst[k] = make_uint2(y[2 * k], y[2 * k + 1]);
                int n2 = 0;  // 16 m
#pragma unroll
                for (int k = 0; k < 6; ++k) n2 = dp4a_ss(y[k], y[k], n2);
                if (mg_lane && r0 + r < rows) {
                    const uint32_t mg = (uint32_t(n2) >> 4) | ((w0[r0 + r] >> 21) & 0x100u);  // g: bit 29 of w0
                    if (WIDTH > 4) *reinterpret_cast<uint16_t*>(mg_at) = uint16_t(mg);
                    else mg_at[0] = uint8_t(mg), mg_at[1] = uint8_t(mg >> 8);
                }
                mg_at += 2u * uint32_t(B);
            }
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kTurns; ++k) {
                const bool second = lane + 32 * k >= kUnits;
                if (unit_at[k] < 24u * uint32_t(cols) && r0 + (second ? 1 : 0) < rows) {
                    int8_t* dst = y_pair + unit_off[k];
                    const unsigned char* src = stage + (lane + 32 * k) * WIDTH;
                    if (WIDTH == 16) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
                    else if (WIDTH == 8) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
                    else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
                }
            }
            y_pair += 2u * row_bytes;
        }
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static int grid_for(size_t items, int threads, int cap) {
    size_t g = (items + threads - 1) / threads;
    if (g > size_t(cap)) g = size_t(cap);
    if (g == 0) g = 1;
    return int(g);
}

cudaError_t launch_decode_file(const void* codes, const void* table, int8_t* y, uint8_t* mg, size_t nblocks,
                               cudaStream_t s) {
    int sms = 0;
    const cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    k_decode_file<<<grid_for(nblocks, 256, sms * 32), 256, 0, s>>>(
        static_cast<const uint8_t*>(codes), static_cast<const DeviceTables*>(table), y, mg, nblocks);
    return cudaGetLastError();
}

cudaError_t launch_pack(const void* codes, const void* table, void* packed, int N, int B, cudaStream_t s) {
    int sms = 0;
    const cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const size_t items = size_t((N + 7) / 8) * ((B + 31) / 32);
    if (items > 0x7FFFFFF0u / 32) return cudaErrorInvalidValue;
    return launch_pdl(k_pack, grid_for(items * 32, 256, sms * 4), 256, 0, s, static_cast<const uint8_t*>(codes),
                      static_cast<const DeviceTables*>(table), static_cast<uint4*>(packed), N, B);
}

cudaError_t launch_decode_packed(const void* packed, const void* table, int8_t* y, uint8_t* mg, int N, int B,
                                 cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const size_t items = size_t((N + 7) / 8) * ((B + 31) / 32);
    if (items > 0x7FFFFFF0u / 32) return cudaErrorInvalidValue;
    constexpr int smem = int(kTableSmemBytes) + kEmitThreads / 32 * kEmitStage;
    static PerDeviceOnce once;
    e = once.run([] {
        auto set = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); };
        cudaError_t r = set(k_decode_packed<16>);
        if (r == cudaSuccess) r = set(k_decode_packed<8>);
        if (r == cudaSuccess) r = set(k_decode_packed<4>);
        return r;
    });
    if (e != cudaSuccess) return e;
    const int grid = grid_for(items * 32, kEmitThreads, sms * 4);
    // every row and every 32 columns (768 bytes) must keep the alignment; a block count that is odd leaves 8
    const bool mg_even = reinterpret_cast<uintptr_t>(mg) % 2 == 0;
    const uintptr_t at = reinterpret_cast<uintptr_t>(y);
    auto kernel = mg_even && at % 16 == 0 && B % 2 == 0 ? k_decode_packed<16> : (mg_even && at % 8 == 0 ? k_decode_packed<8> : k_decode_packed<4>);
    return launch_pdl(kernel, grid, kEmitThreads, smem, s, static_cast<const uint4*>(packed), static_cast<const DeviceTables*>(table), y,
                      mg, N, B);
}

}  // namespace tetra
