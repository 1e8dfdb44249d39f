// Pieces shared by the decode-and-multiply kernels: the lane's activation record, the per-block
// product, the warp's transpose reduction, and the launch helpers.
#pragma once
#include <cuda_fp16.h>

#include "tetra_device.cuh"
#include "tetra_launch.h"

namespace tetra {

constexpr int kRedStride = 36;                 // floats per row of the transpose buffer (32 + pad)
constexpr int kRedFloats = 8 * kRedStride;     // per warp
constexpr int kXqBytesPerCol = 80;             // 3 planes x 24 bytes, step, spare

struct LaneX {
    uint32_t hi[6];   // bits 23..16 of q (signed), int8 x 4
    uint32_t mid[6];  // bits 15..8 (unsigned)
    uint32_t lo[6];   // bits 7..0 (unsigned)
    float step;       // 2^(E-22)
    using Sums = struct PlaneSums;
};

// The planned list's form (pair_planes): 12 + 6 products instead of three times 6, one operation less to put them together.
// (One launch keeps three planes: its chains are short of other work, and a chain of twelve, or two of six and an addition,
// is 1-2 % slower there on half of the sizes.  The planned list: 790 us with three planes, 783 with two.)
struct LanePairs {
    uint32_t hi[12];  // bits 23..8 of q (signed), int16 x 2
    uint32_t lo[6];   // bits 7..0 (unsigned), int8 x 4
    float step;
    using Sums = struct PairSums;
};
// The planes' sums over a block, and what they come to (-sum y q).
struct PlaneSums {
    int h = 0, m = 0, l = 0;
    __device__ __forceinline__ PlaneSums(const FastBlock& fb, const LaneX& X) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            h = dp4a_ss(fb.y[k], X.hi[k], h);
            m = dp4a_su(fb.y[k], X.mid[k], m);
            l = dp4a_su(fb.y[k], X.lo[k], l);
        }
    }
    __device__ __forceinline__ int value() const { return combine_planes(h, m, l); }
};
struct PairSums {
    int h = 0, l = 0;
    __device__ __forceinline__ PairSums(const FastBlock& fb, const LanePairs& X) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            h = dp2a<true>(X.hi[2 * k + 1], fb.y[k], dp2a<false>(X.hi[2 * k], fb.y[k], h));
            l = dp4a_su(fb.y[k], X.lo[k], l);
        }
    }
    __device__ __forceinline__ int value() const { return combine_planes(h, l); }
};

// An inactive lane keeps whatever planes it has read and contributes exact zeros through its step.
__device__ __forceinline__ void lane_x_from_words(const uint32_t q[20], bool active, LaneX& X) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        X.hi[k] = q[k];
        X.mid[k] = q[6 + k];
        X.lo[k] = q[12 + k];
    }
    X.step = active ? __uint_as_float(q[18]) : 0.f;
}

// One block: device word -> contribution scale_b * sum_j y_j x_j (Eq. (2) without
// the row scale).
template <bool HI, typename LX>
__device__ __forceinline__ float block_value(uint32_t sm_tab, uint32_t w0, uint32_t w1pair, const LX& X,
                                             float addend = 0.f) {
    FastBlock fb;
    fast_decode<HI>(sm_tab, w0, w1pair, fb);
    const typename LX::Sums sums(fb, X);
    const float scale = lds32f(scale_address(fb));
    // addend: the caller's running sum (one FFMA)
    return fmaf(float(sums.value()), scale * X.step, addend);
}

// The blocks of one 48-byte record (rows 8G..8G+7 of one column), added to the caller's running sums.  R = 4: half
// a record, the four w0 words in `a` and the two w1 words in h.x, h.y.
template <int R, typename LX>
__device__ __forceinline__ void record_accumulate(uint32_t sm_tab, const uint4& a, const uint4& b, const uint4& h,
                                                  const LX& X, float (&acc)[R]) {
    acc[0] = block_value<false>(sm_tab, a.x, h.x, X, acc[0]);
    acc[1] = block_value<true>(sm_tab, a.y, h.x, X, acc[1]);
    acc[2] = block_value<false>(sm_tab, a.z, h.y, X, acc[2]);
    acc[3] = block_value<true>(sm_tab, a.w, h.y, X, acc[3]);
    if constexpr (R == 8) {
        acc[4] = block_value<false>(sm_tab, b.x, h.z, X, acc[4]);
        acc[5] = block_value<true>(sm_tab, b.y, h.z, X, acc[5]);
        acc[6] = block_value<false>(sm_tab, b.z, h.w, X, acc[6]);
        acc[7] = block_value<true>(sm_tab, b.w, h.w, X, acc[7]);
    }
}
// The same, on their own.
template <int R, typename LX>
__device__ __forceinline__ void record_values(uint32_t sm_tab, const uint4& a, const uint4& b, const uint4& h,
                                              const LX& X, float (&v)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = 0.f;
    record_accumulate<R>(sm_tab, a, b, h, X, v);
}

// Sums v[r] over the 32 lanes for r = 0..7 through the warp's shared-memory
// buffer.  Afterwards lane l holds, for row l / 4, the partial sum over lanes
// 8 (l % 4) .. 8 (l % 4) + 7; the caller finishes with two shuffles.
__device__ __forceinline__ float transpose_partial(float* red, int lane, const float v[8]) {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 8; ++r) red[r * kRedStride + lane] = v[r];
    __syncwarp();
    const float4 s0 = *reinterpret_cast<const float4*>(red + (lane >> 2) * kRedStride + 8 * (lane & 3));
    const float4 s1 = *reinterpret_cast<const float4*>(red + (lane >> 2) * kRedStride + 8 * (lane & 3) + 4);
    return ((s0.x + s0.y) + (s0.z + s0.w)) + ((s1.x + s1.y) + (s1.z + s1.w));
}

// Launch with programmatic stream serialization allowed: the kernel may start while its predecessor
// in the stream is still running and synchronises with it through pdl_wait().
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(unsigned(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}


}  // namespace tetra
