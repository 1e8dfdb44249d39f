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
// in flight.  12288 x 4096: 13.8 us with the map and a row permutation read through L1 and three 2-byte loads,
// now 10.8 us.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 4) k_pack(const uint8_t* __restrict__ codes,
                                                 const DeviceTables* __restrict__ tab,
                                                 uint4* __restrict__ packed, int N, int B) {
    __shared__ uint16_t abx[4096];
    pdl_release();
    for (int i = threadIdx.x; i < 512; i += blockDim.x)
        reinterpret_cast<uint4*>(abx)[i] = __ldg(reinterpret_cast<const uint4*>(tab->trellis_to_abx) + i);
    __syncthreads();
    pdl_wait();  // the words may come from, the packed matrix be read by, the kernel before
    const int groups = (N + 7) / 8, lane = threadIdx.x & 31;
    const int col_groups = (B + 31) / 32, items = groups * col_groups;
    for (int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += (gridDim.x * blockDim.x) >> 5) {
        const int G = it / col_groups, c = min((it - G * col_groups) * 32 + lane, B - 1);
        // a word is 2-byte aligned: its 4-byte aligned part (first or last four bytes) and the other two bytes
        uint32_t four[8], two[8];
        bool front[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint8_t* at = codes + (size_t(min(8 * G + r, N - 1)) * B + c) * 6;
            front[r] = (reinterpret_cast<uintptr_t>(at) & 2) == 0;
            four[r] = __ldg(reinterpret_cast<const uint32_t*>(at + (front[r] ? 0 : 2)));
            two[r] = __ldg(reinterpret_cast<const unsigned short*>(at + (front[r] ? 4 : 0)));
        }
        uint32_t w0[8], w1[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint64_t w = front[r] ? uint64_t(four[r]) | (uint64_t(two[r]) << 32) : uint64_t(two[r]) | (uint64_t(four[r]) << 16);
            file_to_device_word(w, abx[trellis_path(w)], &w0[r], &w1[r]);
            if (8 * G + r >= N) w0[r] = w1[r] = 0u;  // padding rows: the all-zero device word
        }
        if ((it - G * col_groups) * 32 + lane >= B) continue;
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
// through shared memory, so that they leave as contiguous 8-byte stores (a lane's 24 bytes, stored word by word,
// touch every sector six times).  Bound by instruction issue (decoder and byte arithmetic), the stores close behind.
// 12288 x 4096: 35.8 us with direct stores, now 18.9 us (67 MB).
// ---------------------------------------------------------------------------
constexpr int kEmitRows = 2;  // rows decoded and staged at a time (four CTAs then share an SM)
constexpr int kEmitThreads = 256;

// Coordinates of a block in file order, four int8 per word, from the decoder's -8 y.
__device__ __forceinline__ void file_order(const FastBlock& fb, uint32_t (&out)[6]) {
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t v[2];  // y of coordinates 2, 6, 3, 7 and 0, 4, 1, 5
#pragma unroll
        for (int k = 0; k < 2; ++k)  // 16 - y = the five-bit -y with its sign bit flipped; bytes never borrow
            v[k] = (0x90909090u - (((fb.y[2 * s + k] >> 3) & 0x1F1F1F1Fu) ^ 0x10101010u)) ^ 0x80808080u;
        out[2 * s] = prmt(v[1], v[0], 0x6420u);
        out[2 * s + 1] = prmt(v[1], v[0], 0x7531u);
    }
}

template <bool WIDE>
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
    unsigned char* stage = base + kFastBytes + warp * (kEmitRows * 768);
    const int groups = (N + 7) / 8, col_groups = (B + 31) / 32, items = groups * col_groups;
    const int stride = (gridDim.x * blockDim.x) >> 5;
    int it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    uint4 lo, hi, w1;
    auto load = [&](int item) {
        const int G = item / col_groups, c0 = (item - G * col_groups) * 32;
        const uint4* rec = packed + size_t(G) * 3 * B + min(c0 + lane, B - 1);
        lo = __ldg(rec);
        hi = __ldg(rec + B);
        w1 = __ldg(rec + 2 * size_t(B));
    };
    if (it < items) load(it);
    for (; it < items; it += stride) {
        const int G = it / col_groups, c0 = (it - G * col_groups) * 32, cols = min(32, B - c0);
        const uint32_t w0[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        const uint32_t w1p[4] = {w1.x, w1.y, w1.z, w1.w};
        if (it + stride < items) load(it + stride);
#pragma unroll
        for (int r0 = 0; r0 < 8; r0 += kEmitRows) {
            __syncwarp();  // the staged rows of the turn before have been read
            uint32_t mg[kEmitRows];
#pragma unroll
            for (int r = 0; r < kEmitRows; ++r) {
                FastBlock fb;
                if (r & 1) fast_decode<true>(sm_tab, w0[r0 + r], w1p[(r0 + r) >> 1], fb);
                else fast_decode<false>(sm_tab, w0[r0 + r], w1p[(r0 + r) >> 1], fb);
                uint32_t y[6];
                file_order(fb, y);
                uint2* dst = reinterpret_cast<uint2*>(stage + r * 768 + lane * 24);
#pragma unroll
                for (int k = 0; k < 3; ++k) dst[k] = make_uint2(y[2 * k], y[2 * k + 1]);
                int n2 = 0;  // 16 m
#pragma unroll
                for (int k = 0; k < 6; ++k) n2 = dp4a_ss(y[k], y[k], n2);
                mg[r] = (uint32_t(n2) >> 4) | ((w0[r0 + r] >> 17) & 0x100u);  // g: bit 25 of w0
            }
            __syncwarp();
            const int rows = min(kEmitRows, N - 8 * G - r0);
            const size_t block0 = size_t(8 * G + r0) * B + c0;
            if (mg_out && lane < cols) {
#pragma unroll
                for (int r = 0; r < kEmitRows; ++r) {
                    uint8_t* dst = mg_out + 2 * (block0 + size_t(r) * B + lane);
                    if (r < rows) {
                        if (WIDE) *reinterpret_cast<uint16_t*>(dst) = uint16_t(mg[r]);
                        else dst[0] = uint8_t(mg[r]), dst[1] = uint8_t(mg[r] >> 8);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < kEmitRows; ++r) {
                const uint2* src = reinterpret_cast<const uint2*>(stage + r * 768);
                int8_t* dst = y_out + (block0 + size_t(r) * B) * 24;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int i = lane + 32 * k;
                    if (r < rows && i < 3 * cols) {
                        const uint2 v = src[i];
                        if (WIDE) {
                            reinterpret_cast<uint2*>(dst)[i] = v;
                        } else {
                            reinterpret_cast<uint32_t*>(dst)[2 * i] = v.x;
                            reinterpret_cast<uint32_t*>(dst)[2 * i + 1] = v.y;
                        }
                    }
                }
            }
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
    k_decode_file<<<grid_for(nblocks, 256, 148 * 32), 256, 0, s>>>(
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
    constexpr int smem = int(kTableSmemBytes) + kEmitThreads / 32 * kEmitRows * 768;
    static PerDeviceOnce once;
    e = once.run([] {
        cudaError_t r = cudaFuncSetAttribute(k_decode_packed<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r == cudaSuccess) r = cudaFuncSetAttribute(k_decode_packed<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return r;
    });
    if (e != cudaSuccess) return e;
    const int grid = grid_for(items * 32, kEmitThreads, sms * 4);
    const bool wide = reinterpret_cast<uintptr_t>(y) % 8 == 0 && reinterpret_cast<uintptr_t>(mg) % 2 == 0;
    return launch_pdl(wide ? k_decode_packed<true> : k_decode_packed<false>, grid, kEmitThreads, smem, s,
                      static_cast<const uint4*>(packed), static_cast<const DeviceTables*>(table), y, mg, N, B);
}

}  // namespace tetra
