// Decode-and-multiply kernels (Eq. (2), Sec. 5.1) for sm_100a.
//
//   k_gemv_paper  the thread layout the paper describes for its own GPU: a warp
//                 per output row, a lane per block, the six table loads of
//                 Fig. "decode", FP32 multiply-accumulate, shuffle reduction.
//                 Kept as a comparison arm and cross-check.
//   k_gemv_units  the B200 design (also in k_gemv_list, tetra_list.cu): a lane owns one block column and keeps its
//                 24 activations in registers as 24-bit fixed point (here an int16 and
//                 an int8 plane, in k_gemv_list three int8 planes; power-of-two step per
//                 block column, so float16 inputs
//                 within 2^12 of the column's largest are held exactly); it
//                 walks the rows, decodes each word into packed int8 with table
//                 lookups and exclusive ors and multiplies with DP2A and DP4A: products and the sum over
//                 a block are exact integers, one rounding when the block's sum
//                 becomes a float, FP32 accumulation across blocks.  The ALU
//                 pipe only unpacks fields; the integer-MAD pipe does the
//                 arithmetic.
//                 k_gemv_units serves a planned list of matrices from one
//                 persistent grid: k_prepare_x first writes the fixed-point
//                 activations of every matrix to the plan's scratch area, then
//                 every warp walks its own range of passes (32 columns of eight
//                 rows), which may begin and end inside a unit (up to 24 rows of
//                 one matrix, all columns); the last of the warps that share a
//                 unit adds their sums, and no warp ever waits for another.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "tetra_gemv_common.cuh"

namespace tetra {

cudaError_t device_sms(int* sms) {
    static std::mutex mu;
    static int cached[64] = {0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (cached[dev] == 0) {
        int n = 0;
        e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        cached[dev] = n;
    }
    *sms = cached[dev];
    return cudaSuccess;
}

// ===========================================================================
// Paper-design kernel
// ===========================================================================
constexpr int kPaperTile = 64;  // blocks of x per shared-memory tile (the paper's T)

__global__ void __launch_bounds__(256) k_gemv_paper(const uint8_t* __restrict__ codes, size_t row_stride,
                                                    const float* __restrict__ row_scales,
                                                    const DeviceTables* __restrict__ tab,
                                                    const __half* __restrict__ x, float* __restrict__ y, int N, int K,
                                                    int B, int ntail, const __half* __restrict__ tail) {
    __shared__ PaperTables T;
    __shared__ float gain[2];
    __shared__ float xt[kPaperTile * 24];
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&tab->paper);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&T);
        for (int i = threadIdx.x; i < int(sizeof(PaperTables) / 4); i += blockDim.x) dst[i] = src[i];
        if (threadIdx.x < 2) gain[threadIdx.x] = tab->gain[threadIdx.x];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x * 8 + warp;
    const __half* xb = x + size_t(blockIdx.y) * K;
    float acc = 0.f;
    for (int tile0 = 0; tile0 < B; tile0 += kPaperTile) {
        __syncthreads();
        for (int i = threadIdx.x; i < kPaperTile * 24; i += blockDim.x) {
            const int k = tile0 * 24 + i;
            xt[i] = k < K ? __half2float(xb[k]) : 0.f;
        }
        __syncthreads();
        if (row < N) {
            const int end = min(B, tile0 + kPaperTile);
            for (int b = tile0 + lane; b < end; b += 32) {
                int yv[24], m, g;
                decode_file_word(&T, load_file_word(codes + size_t(row) * row_stride, size_t(b)), yv, &m, &g);
                const float* xs = xt + (b - tile0) * 24;
                float dot = 0.f;
#pragma unroll
                for (int j = 0; j < 24; ++j) dot = fmaf(float(yv[j]), xs[j], dot);
                acc = fmaf(gain[g] * T.rsqrt16m[m], dot, acc);
            }
        }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (row < N && lane == 0) {
        float res = row_scales[row] * acc;
        for (int t = 0; t < ntail; ++t)
            res = fmaf(__half2float(tail[size_t(row) * ntail + t]), __half2float(xb[24 * B + t]), res);
        y[size_t(blockIdx.y) * N + row] = res;
    }
}

cudaError_t launch_gemv_paper(const void* codes, size_t row_stride, const float* row_scales, const void* table,
                              const void* x, float* y, int N, int K, int batch, const void* tail, cudaStream_t s) {
    const int ntail = tail ? K % 24 : 0;
    const int B = tail ? K / 24 : (K + 23) / 24;
    dim3 grid((N + 7) / 8, batch);
    k_gemv_paper<<<grid, 256, 0, s>>>(static_cast<const uint8_t*>(codes), row_stride, row_scales,
                                      static_cast<const DeviceTables*>(table), static_cast<const __half*>(x), y, N, K,
                                      B, ntail, static_cast<const __half*>(tail));
    return cudaGetLastError();
}

// ===========================================================================
// Planned list of matrices: k_prepare_x + k_gemv_units
// ===========================================================================
// Workspace, written by grouped_plan (the plan, up to the first pad) and by the kernels:
//   PlanHeader | Problem[count] | unit_prefix[count + 1] | col_prefix[count + 1] | WarpCut[ranges + 1] (optional) | col_start[]
//              | pad | counters | partial sums | pad | xq records
// A unit is groups_per_unit(B) consecutive row groups of one matrix, all columns; a pass is 32 of its columns (or the joint
// pass over its row groups' last, partial column groups).
struct PlanHeader {
    int32_t count;
    int32_t total_units;  // sum over matrices of their units
    int32_t total_cols;   // sum over matrices of words per row, each rounded up to 32 if `aligned`
    int32_t aligned;      // (where the workspace has room for that)
    int32_t row_groups;   // of a unit, at most
    int32_t nwarps;       // warps of the grid that the ranges were cut for (0: no ranges, units are dealt round-robin)
    int32_t warps_per_cta;  // warps of a CTA that have a range
    uint32_t off_problems, off_unit_prefix, off_col_prefix, off_xq;
    uint32_t off_cuts, off_col_start;
    int32_t col_shift;      // col_start names the matrix of every 2^col_shift-th column of the list
    uint32_t off_counters;  // int32 per unit or per range, whichever are fewer: pieces of the cut unit that have arrived
    int32_t counters;
    uint32_t off_partials;  // float [slot][8]: a cut unit's row sums, a slot per piece and row group
    // units [0, dyn_start) are cut into the warps' ranges; the units from
    // dyn_start on are claimed one at a time through dyn_next by warps that have finished their range
    // (k_prepare_x sets dyn_next = dyn_start before every run)
    int32_t dyn_start;
    int32_t dyn_matrix;  // matrix of unit dyn_start
    int32_t dyn_next;
};
constexpr int kDynamicTailPermille = 100;  // share of the list's work left for the claimed units
constexpr int kClaimPasses = 128;          // passes per warp from which on there are claimed units (see cut_ranges)
// What the ranges are cut by: a pass, and a row group's fold, row scales and tail.  (With two per unit instead of four per row
// group the warps that have units of one row group, 16 passes each, finished 8 % before those with units of three.)
constexpr int kPassCost = 8, kFoldCost = 4;

// Where a warp's range begins; the next entry is where it ends.  A range that begins inside a unit (pass > 0) shares that
// unit with the ranges before it: `pieces` ranges in all, of which the first, the one in which the unit begins, is `back` ranges
// before this one; `slot` is the unit's first.  (Twelve bytes: the cuts for 160 multiprocessors have to lie in the 32 KB that
// the workspace has always had for them.)
struct WarpCut {
    int32_t unit;
    uint32_t at;     // matrix of the unit << 8 | pass
    uint32_t piece;  // slot << 16 | pieces << 8 | back
    __device__ __host__ static int pass(uint32_t at) { return int(at & 255u); }
    __device__ __host__ static int matrix(uint32_t at) { return int(at >> 8); }
};
constexpr int kMaxUnitPasses = 3 * 63 + 1;  // (more than one row group: at most ten columns beside full groups, 2048 columns)
static_assert(kMaxUnitPasses < 256, "a pass, and the pieces of a unit, in eight bits");

static inline int problem_blocks(const Problem& q) {
    return (q.tail || q.K % 24 == 0) ? q.K / 24 : (q.K + 23) / 24;
}

// Row groups (of eight rows) one unit covers.  When the last column group of a matrix is at most
// half full (B mod 32 in 1..16), up to three consecutive row groups share one pass over it, so that
// pass runs with most lanes busy instead of B mod 32 of them.
constexpr int kMaxRowGroups = 3;
__host__ __device__ inline int groups_per_unit(int B, int most) {
    const uint32_t rem = uint32_t(B) & 31u;
    const int r = rem - 1u < 10u ? 3 : (rem - 1u < 16u ? 2 : 1);
    return r < most ? r : most;
}
static inline int problem_units(const Problem& q, int row_groups) {
    const int R = groups_per_unit(problem_blocks(q), row_groups);
    return ((q.N + 7) / 8 + R - 1) / R;
}

// k_gemv_units keeps the places of a matrix's records as 16-byte units in 32 bits (in 64 bits a pass of the 8B model takes 770
// to 775 us instead of 765).  A matrix that is larger is planned as slices of this many rows: problems of their own, one behind
// the other, that share their activation records.
static inline long long slice_rows(const Problem& q) { return 8 * (0xFFFFFFFELL / (3 * problem_blocks(q)) / 6 * 6); }
int problem_slices(const Problem& q) {
    if ((q.N + 7LL) / 8 * 3 * problem_blocks(q) < 0x80000000LL) return 1;
    return int((q.N + slice_rows(q) - 1) / slice_rows(q));
}
Problem problem_slice(const Problem& q, int i) {
    const long long rows = slice_rows(q), row0 = i * rows;
    Problem p = q;
    p.codes = static_cast<const char*>(q.codes) + row0 / 8 * 48 * problem_blocks(q);
    p.row_scales = q.row_scales + row0;
    if (q.tail) p.tail = static_cast<const char*>(q.tail) + 2 * row0 * (q.K % 24);
    p.y = q.y + row0;
    p.N = int32_t(q.N - row0 < rows ? q.N - row0 : rows);
    return p;
}
// b is the slice behind a: its columns are a's
static inline bool same_columns(const Problem& a, const Problem& b) {
    return b.x == a.x && b.K == a.K && !b.tail == !a.tail && a.N == slice_rows(a) &&
           b.codes == static_cast<const char*>(a.codes) + (long long)(a.N / 8) * 48 * problem_blocks(a);
}

// The activation records of 32 columns lie together, part by part: 16 bytes of every column, then the next 16.  A warp's load
// is then 512 contiguous bytes, four wavefronts, and not 32 pieces 80 bytes apart (8B pass 773 -> 763 us, one layer of it
// 34.7 -> 32.7).  In a plan whose columns are not aligned a column's 80 bytes lie together and a matrix takes no more than
// those (the same times and 769.6 us, 35.9 us with them).
static inline long long problem_cols(const Problem& q, bool aligned) {
    const int B = problem_blocks(q);
    return aligned ? (B + 31) & ~31 : B;
}
template <bool ALIGNED>
__device__ __forceinline__ uint32_t record_at(uint32_t col) {
    constexpr uint32_t U = kXqBytesPerCol / 16;
    return ALIGNED ? (col >> 5) * (32 * U) + (col & 31u) : col * U;
}

// Bytes of a plan: what the kernels read, and what they keep beside it.
static size_t plan_meta_bytes(int count, int ranges, int starts) {
    const size_t b = sizeof(PlanHeader) + size_t(count) * sizeof(Problem) + 2 * size_t(count + 1) * 4 +
                     (ranges ? size_t(ranges + 1) * sizeof(WarpCut) : 0) + size_t(starts) * 4;
    return (b + 255) & ~size_t(255);
}
static size_t plan_bytes(size_t meta, int counters, size_t slots, size_t cols) {
    return ((meta + size_t(counters) * 4 + slots * 32 + 127) & ~size_t(127)) + cols * kXqBytesPerCol;
}
// Entries of col_start: a column in 64, but no more than four a matrix.
static int col_shift_for(size_t cols, int count) {
    int shift = 6;
    while ((cols >> shift) + 1 > 4 * size_t(count)) ++shift;
    return shift;
}

// What a caller is asked for.  A list of at most kRoomTasks (row group, column group) pairs is given 32 bytes a pair, which hold
// the pieces of any cut of units of one row group.  A longer one is given six slots a range and room for aligned columns (where
// that is less than a sixteenth of its codes), but planned without them too: callers may have a workspace of a fixed size, and
// these were not always asked for (8B, 4 / 8 / 12 / 36 layers 97 / 181 / 263 / 754 us, in the smaller workspace 117 / 195 /
// 274 / 781).
constexpr long long kRoomTasks = 65536;
constexpr size_t kCutsRoom = 8193 * 4, kMatrixRoom = 16, kRangesRoom = 2560;  // (2560 ranges: 160 multiprocessors)
static_assert((kRangesRoom + 1) * sizeof(WarpCut) + sizeof(PlanHeader) - 56 < kCutsRoom, "the cuts have room");
static size_t workspace_bytes(const Problem* problems, int count, bool room_of_long_lists) {
    size_t cols = 0, groups = 0, tasks = 0, blocks = 0, padding = 0;
    for (int i = 0; i < count; ++i) {
        const size_t B = size_t(problem_blocks(problems[i])), G = (size_t(problems[i].N) + 7) / 8;
        cols += B;
        padding += (32 - B % 32) % 32 * kXqBytesPerCol;
        blocks += G * B;
        groups += G;
        tasks += G * ((B + 31) / 32);
    }
    size_t b = (56 + size_t(count) * (sizeof(Problem) + kMatrixRoom) + 2 * size_t(count + 1) * 4 + kCutsRoom + 255) & ~size_t(255);
    b += cols * kXqBytesPerCol;
    if (tasks <= size_t(kRoomTasks)) b = ((b + 255) & ~size_t(255)) + groups * 4 + 256 + tasks * 32;
    else if (room_of_long_lists) b += kRangesRoom * (4 + 6 * 32) + (padding <= 3 * blocks ? padding + 256 : 0);
    return b;
}
size_t grouped_workspace_bytes(const Problem* problems, int count) { return workspace_bytes(problems, count, true); }
size_t grouped_workspace_least(const Problem* problems, int count) { return workspace_bytes(problems, count, false); }

// One thread per column of the list.  What bounds it is a chain of dependent loads; a column's matrix is named by the plan
// instead of searched for.  The plan may come from the kernel before (tetra_gemv_noalloc writes one, a caller may have copied
// it), so nothing of it is read ahead of the wait; and k_gemv_units, which does read it ahead of its own, is released only
// when the grids before this one are complete (8B pass 764.5 us instead of 762.4, one layer of it 34.1 instead of 32.7).
__global__ void __launch_bounds__(128) k_prepare_x(unsigned char* __restrict__ ws) {
    pdl_wait();  // the activations and the plan may come from the previous kernel of the stream
    pdl_release();
    const PlanHeader* H = reinterpret_cast<const PlanHeader*>(ws);
    const Problem* problems = reinterpret_cast<const Problem*>(ws + H->off_problems);
    const int32_t* col_prefix = reinterpret_cast<const int32_t*>(ws + H->off_col_prefix);
    const int32_t* col_start = reinterpret_cast<const int32_t*>(ws + H->off_col_start);
    uint4* xq = reinterpret_cast<uint4*>(ws + H->off_xq);
    const int total = H->total_cols, threads = int(gridDim.x * blockDim.x);
    int gc = blockIdx.x * blockDim.x + threadIdx.x;
    const __half* x = nullptr;
    int K = 0, c = 0, cols = 0, begin = 0;
    const int col_shift = H->col_shift;
    const bool aligned = H->aligned;
    auto find = [&] {
        if (gc >= total) return;
        int p = __ldg(col_start + (gc >> col_shift));
        while (__ldg(col_prefix + p + 1) <= gc) ++p;
        begin = __ldg(col_prefix + p);
        c = gc - begin;
        x = static_cast<const __half*>(problems[p].x);
        K = problems[p].K;
        cols = problems[p].tail ? K / 24 : (K + 23) / 24;
    };
    find();
    for (; gc < total; gc += threads, find()) {
        if (c >= cols) continue;
        uint32_t q[20];
        quantise_column(x, K, c, q);
        pair_planes(q);
        uint4* rec = xq + size_t(begin) * (kXqBytesPerCol / 16) + (aligned ? record_at<true>(uint32_t(c)) : record_at<false>(uint32_t(c)));
        const int part = aligned ? 32 : 1;
#pragma unroll
        for (int k = 0; k < 5; ++k) rec[part * k] = make_uint4(q[4 * k], q[4 * k + 1], q[4 * k + 2], q[4 * k + 3]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0)
        reinterpret_cast<PlanHeader*>(ws)->dyn_next = H->dyn_start;  // the claimed units start over
    int32_t* counters = reinterpret_cast<int32_t*>(ws + H->off_counters);  // and so do the arrivals at cut units
    for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < H->counters; w += threads) counters[w] = 0;
}

// This lane's activation record (global memory, L1/L2 resident) into registers.
template <bool ALIGNED>
__device__ __forceinline__ void load_lane_x(const uint4* src, bool active, LanePairs& X) {
    constexpr int part = ALIGNED ? 32 : 1;
    const uint4 t0 = __ldg(src), t1 = __ldg(src + part), t2 = __ldg(src + 2 * part), t3 = __ldg(src + 3 * part), t4 = __ldg(src + 4 * part);
    X.hi[0] = t0.x; X.hi[1] = t0.y; X.hi[2] = t0.z; X.hi[3] = t0.w; X.hi[4] = t1.x; X.hi[5] = t1.y;
    X.hi[6] = t1.z; X.hi[7] = t1.w; X.hi[8] = t2.x; X.hi[9] = t2.y; X.hi[10] = t2.z; X.hi[11] = t2.w;
    X.lo[0] = t3.x; X.lo[1] = t3.y; X.lo[2] = t3.z; X.lo[3] = t3.w; X.lo[4] = t4.x; X.lo[5] = t4.y;
    X.step = active ? __uint_as_float(t4.z) : 0.f;  // an inactive lane contributes exact zeros
}

#ifndef TETRA_UNIT_THREADS
#define TETRA_UNIT_THREADS 512
#endif
constexpr int kUnitThreads = TETRA_UNIT_THREADS;
constexpr int kUnitWarps = kUnitThreads / 32;
constexpr int kUnitFloats = kRedFloats + 96;  // per warp: the transpose buffer, and a sum per row group and lane

// Every warp walks its range of passes.  wait: for k_prepare_x.
template <bool ALIGNED, typename Wait>
__device__ __forceinline__ void walk_units(unsigned char* __restrict__ ws, unsigned char* smem, uint32_t sm_tab, Wait wait) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* red = reinterpret_cast<float*>(smem + kFastBytes) + warp * kUnitFloats;
    float* sums = red + kRedFloats + lane;  // of row group gi, row lane / 4: this lane's part at 32 gi
    const PlanHeader* H = reinterpret_cast<const PlanHeader*>(ws);
    const Problem* problems = reinterpret_cast<const Problem*>(ws + sizeof(PlanHeader));
    auto unit_prefix = [&](int i) { return __ldg(reinterpret_cast<const int32_t*>(ws + H->off_unit_prefix) + i); };

    // This warp's share: a contiguous range cut for equal work when the plan holds ranges for this
    // grid (neighbouring warps then walk neighbouring row groups of the same matrices), else every
    // (warps in grid)-th unit.
    const int gw = blockIdx.x * kUnitWarps + warp, nw = gridDim.x * kUnitWarps;
    int u = gw, u_end = H->total_units, u_step = nw;
    bool claim = false;  // after the range: claim the units from dyn_start on, one at a time
    int pass0 = 0;       // where in its first unit the range begins
    const WarpCut* cut = nullptr;
    int p = -1, p_begin = 0, p_end = 0;  // matrix of the current unit and its range of units
    // per matrix, kept in registers across its units (everything else is re-read where it is needed: with the row groups in a
    // register too the 8B pass takes 764 us instead of 755, with more of these re-read 774)
    const uint4* codes_p = nullptr;
    uint32_t x_p = 0;                    // its activation records, in 16-byte units from the workspace's first byte
    uint32_t Bu = 1;
    bool have_record = false;            // the ring already holds the first record of the unit about to start
    auto enter_matrix = [&] {
        p_end = unit_prefix(p + 1);
        p_begin = unit_prefix(p);
        const Problem& Q = problems[p];
        const int K = Q.K;
        Bu = uint32_t(Q.tail ? K / 24 : (K + 23) / 24);
        codes_p = static_cast<const uint4*>(Q.codes);
        x_p = (H->off_xq >> 4) + uint32_t(__ldg(reinterpret_cast<const int32_t*>(ws + H->off_col_prefix) + p)) * uint32_t(kXqBytesPerCol / 16);
        have_record = false;
    };
    // Code records reach the decoder through a per-warp ring in shared memory: two slots of 3 x 512
    // bytes (one 16-byte part per lane), filled with cp.async one pass ahead, so the prefetch holds
    // no registers while eight blocks are being decoded.  Each lane reads back only what it copied.
    const uint32_t ring = sm_tab + uint32_t(kFastBytes) + uint32_t(kUnitWarps * kUnitFloats * 4) + uint32_t(warp) * 3072u + uint32_t(lane) * 16u;
    uint32_t slot = ring;                  // of the pass at hand
    const uint32_t slots = 2 * ring + 1536;  // the two slots' sum

    auto request = [&](uint32_t dst, uint32_t at) {  // the three parts of the record at `at`
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(codes_p + at));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + 512), "l"(codes_p + (at + Bu)));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + 1024), "l"(codes_p + (at + 2 * Bu)));
    };
    // This lane's place in the joint pass over the partial column group of a unit's ng row groups: whether it has one, its
    // column, and its record from the unit's first.
    struct Place { bool in; uint32_t col, record; };
    auto joint_place = [&](int ng) {
        const int rem = int(Bu & 31u), group = rem ? min(lane / max(rem, 1), 3) : 0;
        const bool in = rem && group < ng;
        const uint32_t col = (Bu & ~31u) + (in ? uint32_t(lane - group * rem) : 0u);
        return Place{in, col, uint32_t(in ? group : 0) * 3u * Bu + col};
    };
    // ahead of the wait: the plan, and the range's first record (both are older than k_prepare_x, which releases this kernel
    // behind its own wait); with a joint pass's too q, k, v of an 8B layer 13.1 -> 12.9 us
    if (H->nwarps == nw) {
        const bool has_range = warp < H->warps_per_cta;
        u = u_end = H->total_units;
        u_step = 1;
        if (has_range) {
            cut = reinterpret_cast<const WarpCut*>(ws + H->off_cuts) + (blockIdx.x * H->warps_per_cta + warp);
            const uint32_t at = __ldg(&cut[0].at);
            u = __ldg(&cut[0].unit);
            pass0 = WarpCut::pass(at);
            u_end = __ldg(&cut[1].unit) + (WarpCut::pass(__ldg(&cut[1].at)) > 0);
            claim = H->dyn_start < H->total_units;
            if (u < u_end) {
                p = WarpCut::matrix(at);
                enter_matrix();
                const int R = groups_per_unit(int(Bu), H->row_groups), CGf = int(Bu >> 5), g0 = (u - p_begin) * R;
                const int gi = CGf ? pass0 / CGf : 0, ng = min(R, (problems[p].N + 7) / 8 - g0);
                const bool full = CGf && gi < ng;
                request(slot, uint32_t(g0) * 3u * Bu + (full ? uint32_t(gi) * 3u * Bu + uint32_t(lane + 32 * (pass0 - gi * CGf)) : joint_place(ng).record));
                have_record = true;
            }
        }
    }
    asm volatile("cp.async.commit_group;");
    wait();  // the activation records (and zeroed counters) come from k_prepare_x

    for (;; u += u_step) {
        if (u >= u_end) {
            if (!claim) break;
            // The range is done: claim one of the units that were left unassigned.  One atomic per unit; it
            // only hands out numbers, nothing waits on it, and the numbers a warp gets increase, so the walk
            // below still only goes up.  (Claiming one unit ahead would hide the atomic's latency but keeps a
            // register live across the passes, which costs more than it saves.)
            int c = 0;
            if (lane == 0) c = atomicAdd(&reinterpret_cast<PlanHeader*>(ws)->dyn_next, 1);
            c = __shfl_sync(0xFFFFFFFFu, c, 0);
            if (c >= H->total_units) break;
            u = c;
            u_end = c + 1;
            if (p < H->dyn_matrix) p_end = 0, p = H->dyn_matrix - 1;
            cut = nullptr;  // (the last range ends where the first of these units begins)
            have_record = false;
        }
        if (u >= p_end) {  // first unit, or the walk has left the matrix: units only go up
            do ++p; while (u >= unit_prefix(p + 1));
            enter_matrix();
        }
        const int CGf = int(Bu >> 5);   // full column groups
        const int rem = int(Bu & 31);   // columns of the last, partial one
        const int R = groups_per_unit(int(Bu), H->row_groups);
        const int g0 = (u - p_begin) * R;
        const int ng = min(R, (problems[p].N + 7) / 8 - g0);
        const Place place = joint_place(ng);
        const bool lane_in = place.in;
        const uint32_t lane_col = place.col;
        const bool next_unit_here = CGf > 0 && u + u_step < min(u_end, p_end);

        // the passes of this unit that the range holds: all of them, unless the range begins or ends inside it
        int left = ng * CGf + (rem > 0);
        const bool ends_inside = cut && u == __ldg(&cut[1].unit);  // (a range that ends between two units does not reach the second)
        if (ends_inside) left = WarpCut::pass(__ldg(&cut[1].at));
        left -= pass0;
        bool joint = pass0 >= ng * CGf;
        int gi = joint ? 0 : pass0 / CGf;
        const int cg0 = pass0 - gi * CGf;
        const uint32_t unit0 = uint32_t(g0) * 3u * Bu + uint32_t(lane), unit_rem = uint32_t(g0) * 3u * Bu + place.record;
        // places are kept as 16-byte units from the matrix's first record, in 32 bits
        uint32_t record = joint ? unit_rem : unit0 + uint32_t(gi) * 3u * Bu + 32u * uint32_t(cg0);  // of the pass at hand

        if (!have_record) {
            request(slot, record);
            asm volatile("cp.async.commit_group;");
        }
        sums[0] = sums[32] = sums[64] = 0.f;
        {   // row scales and tails of the unit, which its end would wait for (8B pass 781 -> 773 us)
            const Problem& Q = problems[p];
            const int row0 = 8 * g0, rows = min(8 * ng, Q.N - row0), ntail = Q.tail ? Q.K % 24 : 0;
            if (ntail && 128 * lane < 2 * rows * ntail + 127) {
                const char* at = static_cast<const char*>(Q.tail) + 2 * size_t(row0) * ntail;
                asm volatile("prefetch.global.L1 [%0];" :: "l"(at + min(128 * lane, 2 * rows * ntail - 1)));
            }
            if (lane == 31) asm volatile("prefetch.global.L1 [%0];" :: "l"(Q.row_scales + row0));
        }
        float acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r] = 0.f;

        // One pass = one 48-byte record per lane: the full column groups of each row group in turn, then the joint pass over
        // the partial column group (a single call site of the decoder).  A segment is a row group's full column groups, or
        // the joint pass: inside one, records and activations follow at fixed distances.
        bool lane_on = !joint || lane_in;
        int seg = joint ? 1 : min(CGf - cg0, left);                        // passes left in the segment
        left -= seg;                                                       // and behind it
        uint32_t x_at = x_p + record_at<ALIGNED>(joint ? lane_col : uint32_t(lane + 32 * cg0));
        // the first record behind the segment: the next row group's, the joint pass's, the next unit's
        constexpr uint32_t kNone = 0xFFFFFFFFu;
        auto behind = [&]() -> uint32_t {
            if (left) return gi + 1 < ng ? unit0 + uint32_t(gi + 1) * 3u * Bu : unit_rem;
            return next_unit_here ? unit0 + uint32_t(u_step * R) * 3u * Bu : kNone;
        };
        uint32_t after = behind();
        for (;;) {
            uint4 a, b, h;
            {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w) : "r"(slot));
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "r"(slot + 512));
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(h.x), "=r"(h.y), "=r"(h.z), "=r"(h.w) : "r"(slot + 1024));
            }
            slot = slots - slot;
            // ahead of the next record's copies: the same unit serves both in order, and a load behind a copy waits for
            // memory (Qwen3-8B pass 810 -> 803 us)
            LanePairs X;
            load_lane_x<ALIGNED>(reinterpret_cast<const uint4*>(ws) + x_at, lane_on, X);
            x_at += 32 * kXqBytesPerCol / 16;
            // prefetch the next pass's record (or the first one of this warp's next unit)
            record = seg == 1 ? after : record + 32u;
            if (record != kNone) request(slot, record);
            asm volatile("cp.async.commit_group;");
            record_accumulate<8>(sm_tab, a, b, h, X, acc);  // acc is zero when a segment begins
            if (--seg) continue;
            if (joint) {
                // lane -> (row group, column); lane l then sums, for row l / 4, the columns
                // k = l % 4, l % 4 + 4, ... of every row group's segment of the buffer
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 8; ++r) red[r * kRedStride + lane] = acc[r];
                __syncwarp();
                const float* rr = red + (lane >> 2) * kRedStride;
                float s0 = sums[0], s1 = sums[32], s2 = sums[64];
                for (int k = lane & 3; k < rem; k += 4) {
                    s0 += rr[k];
                    if (R > 1) s1 += rr[rem + k];
                    if (R > 2) s2 += rr[2 * rem + k];
                }
                sums[0] = s0;
                sums[32] = s1;
                sums[64] = s2;
                break;
            }
            // row group done: fold its eight accumulators into this lane's row
            sums[32 * gi] = transpose_partial(red, lane, acc);
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r] = 0.f;
            if (!left) break;
            ++gi;
            x_at = x_p + record_at<ALIGNED>(uint32_t(lane));
            seg = min(CGf, left);
            if (gi == ng) {
                joint = true;
                lane_on = lane_in;
                seg = 1;
                x_at = x_p + record_at<ALIGNED>(lane_col);
            }
            left -= seg;
            after = behind();
        }
        have_record = next_unit_here;
        // What the end of the unit needs is loaded here: the fence behind a piece empties L1, and what is read behind it waits for
        // L2 one load after the other (1024 x 4096 8.5 -> 8.3 us, 8B pass 766 -> 760).
        const Problem& Q = problems[p];
        const int N = Q.N, ntail = Q.tail ? Q.K % 24 : 0, row0 = 8 * g0 + (lane >> 2);
        const __half *tails = static_cast<const __half*>(Q.tail), *xh = static_cast<const __half*>(Q.x) + 24 * Bu;
        float* y = Q.y;
        float scale[kMaxRowGroups];
#pragma unroll
        for (int k = 0; k < kMaxRowGroups; ++k) scale[k] = k < ng && row0 + 8 * k < N ? __ldg(Q.row_scales + row0 + 8 * k) : 0.f;
        // A unit that other ranges share: this range's piece goes to the workspace, and the last piece to arrive finds the
        // others there (a counter, nothing waits on it) and adds them in the ranges' order.
        const WarpCut* shared = pass0 ? cut : (ends_inside ? cut + 1 : nullptr);
        pass0 = 0;
        if (shared) {
            const uint32_t info = __ldg(&shared->piece);
            const int range = blockIdx.x * H->warps_per_cta + warp;
            const int pieces = int(info >> 8 & 255u), first = range + int(shared - cut) - int(info & 255u);
            float* all = reinterpret_cast<float*>(ws + H->off_partials) + size_t(info >> 16) * 8 + (lane >> 2);
            float* mine = all + (range - first) * ng * 8;
            const uint32_t counter = H->off_counters + 4u * uint32_t(H->counters == H->total_units ? u : first);
#pragma unroll
            for (int k = 0; k < kMaxRowGroups; ++k) {
                float v = sums[32 * k];
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
                if ((lane & 3) == 0 && k < ng) __stcg(mine + 8 * k, v);
            }
            __threadfence();
            __syncwarp();
            int arrived = 0;
            if (lane == 0) arrived = atomicAdd(reinterpret_cast<int32_t*>(ws + counter), 1);
            if (__shfl_sync(0xFFFFFFFFu, arrived, 0) != pieces - 1) continue;
            __threadfence();
            float s0 = 0.f, s1 = 0.f, s2 = 0.f;
            if (ng == 1) {
#pragma unroll 4
                for (int k = lane & 3; k < pieces; k += 4) s0 += __ldcg(all + 8 * k);
            } else {  // (of two row groups the third sum is not read)
                for (int k = lane & 3; k < pieces; k += 4) {
                    const float* theirs = all + k * ng * 8;
                    s0 += __ldcg(theirs);
                    s1 += __ldcg(theirs + 8);
                    if (ng > 2) s2 += __ldcg(theirs + 16);
                }
            }
            sums[0] = s0;
            sums[32] = s1;
            sums[64] = s2;
        }
        // row scale, tail (Sec. 5.1; four lanes per row share the tail), store
#pragma unroll
        for (int gk = 0; gk < kMaxRowGroups; ++gk) {
            if (gk >= ng) break;
            const int row = row0 + 8 * gk;
            float sum = sums[32 * gk] * scale[gk];
            if (row < N) {
                const __half* tl = tails + size_t(row) * ntail;
                for (int k = lane & 3; k < ntail; k += 4) sum = fmaf(__half2float(tl[k]), __half2float(xh[k]), sum);
            }
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 1);
            sum += __shfl_xor_sync(0xFFFFFFFFu, sum, 2);
            if (row < N && (lane & 3) == 0) y[row] = sum;
        }
    }
}

// (Out of line: with both copies in the kernel a pass of the 8B model takes 769 us instead of 764.)
template <typename Wait>
__device__ __noinline__ void walk_unaligned(unsigned char* ws, unsigned char* smem, uint32_t sm_tab, Wait wait) {
    walk_units<false>(ws, smem, sm_tab, wait);
}

// The persistent kernel of a planned list.  All that it needs to know is in the workspace, so a workspace can be copied or moved
// and still runs correctly: the host needs no record of it.
__global__ void __launch_bounds__(kUnitThreads, 1)
k_gemv_units(const DeviceTables* __restrict__ tab, unsigned char* __restrict__ ws) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_release();
    unsigned char* smem = stage_fast_tables(tab, smem_raw);
    const uint32_t sm_tab = smem_u32(smem);
    __syncthreads();  // the only CTA-wide barrier: the tables are staged (by cp.async, the plan read meanwhile: 783 instead of
                      // 773 us for the 8B pass)
    const auto wait = [] { pdl_wait(); };
    if (reinterpret_cast<const PlanHeader*>(ws)->aligned) walk_units<true>(ws, smem, sm_tab, wait);
    else walk_unaligned(ws, smem, sm_tab, wait);
}

// A matrix as the ranges are cut: units of up to R of its G row groups, each of CG full column groups and perhaps a partial one.
struct MatrixUnits {
    int R, G, CG, partial;
    long long units;
    int groups(long long k) const { return int(G - k * R < R ? G - k * R : R); }  // of unit k
    int passes(long long k) const { return groups(k) * CG + partial; }
};

// Cuts the list's passes into the ranges of the grid's warps; `inside`: also inside units.  Returns the slots that the pieces of
// cut units take.
static size_t cut_ranges(PlanHeader* H, const MatrixUnits* M, const int32_t* up, WarpCut* cuts, int sms, bool inside) {
    const int count = H->count;
    const long long units = H->total_units;
    // Cut the sequence of passes into contiguous ranges of equal work.  A cut inside a unit costs its two sides a store of
    // sums and an atomic, two of each per warp and run; cut between units only, a list of a few layers leaves most warps
    // waiting for those with one unit more (4B, one / two / six layers 28.9 / 40.9 / 92.6 us, cut inside units
    // 24.8 / 39.0 / 87.3; 14B, one layer 59.2 and 51.4).
    long long passes = 0;
    for (int i = 0; i < count; ++i) passes += (M[i].units - 1) * M[i].passes(0) + M[i].passes(M[i].units - 1);
    long long per = (passes + sms - 1) / sms;  // warps of a CTA that have a range: no more than passes
    if (per > kUnitWarps) per = kUnitWarps;
    H->warps_per_cta = int32_t(per);
    const int ranges = int(per) * sms;
    // With no more passes than ranges each has its own: cut by cost some warps get two (3072 x 4096 10.1 us instead of 9.6), and a
    // list of few passes begins in a later CTA (64 x 768 5.3 instead of 5.1).
    const bool one_each = inside && passes <= ranges;
    const int fold_cost = one_each ? 0 : kFoldCost;
    auto full_work = [&](int i) { return (long long)M[i].passes(0) * kPassCost + fold_cost * M[i].groups(0); };  // of all units but the last
    auto matrix_work = [&](int i) {
        const long long U = M[i].units;
        return (U - 1) * full_work(i) + M[i].passes(U - 1) * kPassCost + fold_cost * M[i].groups(U - 1);
    };
    long long total = 0;
    for (int i = 0; i < count; ++i) total += matrix_work(i);
    // Of a long list the last tenth of the work is not assigned: warps that finish early claim it unit by unit, which
    // evens out what the cost model and the warps' unequal speeds leave.  A unit claimed last still makes the others wait
    // for it, which shorter lists do not make up for.  All assigned / a tenth claimed, us: 8B, 8 / 12 / 16 / 36 layers
    // 187 / 274 / 360 / 791 and 191 / 269 / 355 / 772; 4B, 10 / 16 / 36 135 / 208 / 451 and 136 / 205 / 434; 14B, 4 /
    // 36 layers 167 / 1436 and 168 / 1375 (7 passes per warp are a layer of the 4B model, 13 of the 8B, 24 of the 14B).
    // 6 % claimed: 8B, 36 layers 785; 15 % 777.  Units claimed while the one before is at work, so that its first record
    // is not waited for: 779 (a warp then holds one more unit at the end); two or three short units at a time: 14B 1410.
    // Cut between units, claimed units also make up for unequal ranges, from eight units per warp on (8B, eight layers 204
    // without and 199 with them; 4B, two layers, 45.5 and 50.2).
    H->dyn_start = int32_t(units);
    const bool claimed = inside ? passes >= (long long)kClaimPasses * H->nwarps : units >= 8LL * H->nwarps;
    if (claimed) {
        const long long planned = total - total * kDynamicTailPermille / 1000;
        long long acc = 0;
        int i = 0;
        while (i < count - 1 && acc + matrix_work(i) <= planned) acc += matrix_work(i++);
        long long ds = up[i] + (planned - acc) / full_work(i);
        if (ds > units) ds = units;
        H->dyn_start = int32_t(ds);
        total = acc + (ds - up[i]) * full_work(i);
    }
    auto matrix_of = [&](int from, long long uu) {
        while (from > 0 && up[from] > uu) --from;
        while (from < count - 1 && up[from + 1] <= uu) ++from;
        return from;
    };
    int pi = 0;
    long long before = 0, work = matrix_work(0), unit_work = full_work(0);  // work of matrices 0..pi-1, of matrix pi, of its units
    const long long step = total / ranges, step_rest = total % ranges;
    long long target = 0, rest = 0;
    for (int w = 0; w < ranges; ++w) {
        if (w) {  // total * w / ranges, in steps
            target += step;
            if ((rest += step_rest) >= ranges) rest -= ranges, ++target;
        }
        if (one_each) target = w < passes ? w * (long long)kPassCost : total;
        while (pi < count - 1 && before + work <= target) {
            before += work;
            work = matrix_work(++pi);
            unit_work = full_work(pi);
        }
        const long long at = target - before;
        const long long k = at >> 32 ? at / unit_work : uint32_t(at) / uint32_t(unit_work);
        long long uu = up[pi] + k, pass = inside ? (at - k * unit_work) / kPassCost : 0;
        if (pass >= M[pi].passes(k)) { pass = 0; ++uu; }
        if (w && inside && !one_each) {
            const WarpCut& last = cuts[w - 1];
            const int last_pass = WarpCut::pass(last.at);
            if (uu < last.unit || (uu == last.unit && pass <= last_pass && last_pass)) {
                // fewer passes than ranges: one pass behind the range before
                uu = last.unit;
                pass = last_pass + 1;
                const int pj = matrix_of(WarpCut::matrix(last.at), uu);
                if (uu >= units || pass >= M[pj].passes(uu - up[pj])) { ++uu; pass = 0; }
            }
        }
        if (uu >= H->dyn_start) { uu = H->dyn_start; pass = 0; }
        // (a cut may have moved on from the matrix that its target lies in, or back from it)
        cuts[w] = WarpCut{int32_t(uu), uint32_t(matrix_of(pi, uu)) << 8 | uint32_t(pass), 0};
    }
    H->dyn_matrix = matrix_of(0, H->dyn_start);
    cuts[ranges] = WarpCut{H->dyn_start, uint32_t(H->dyn_matrix) << 8, 0};
    // who shares a cut unit: the range before the first that begins inside it, and all that begin inside it
    size_t slots = 0;
    for (int w = 1; w < ranges; ++w) {
        if (!WarpCut::pass(cuts[w].at)) continue;
        int last = w;
        while (last + 1 < ranges && cuts[last + 1].unit == cuts[w].unit) ++last;
        const int i = WarpCut::matrix(cuts[w].at), pieces = last - w + 2;
        for (int v = w; v <= last; ++v) cuts[v].piece = uint32_t(slots) << 16 | uint32_t(pieces) << 8 | uint32_t(v - w + 1);
        slots += size_t(pieces) * M[i].groups(cuts[w].unit - up[i]);
        w = last;
    }
    H->counters = slots ? int32_t(units < ranges ? units : ranges) : 0;
    return slots;
}

// The plan of a list for a grid of `sms` CTAs in ws_bytes of workspace: its first `meta` bytes, allocated.  Of these the first
// that has room: ranges cut inside units of up to three row groups, inside units of one, between units, which takes no slots; no
// ranges; and of each with aligned columns or without.  A list with at most two (row group, column group) pairs per warp
// begins with the second: a piece for each pair, 6 of a row group of 4096 columns instead of 16 of a unit (units of three and of
// one: 1024 x 2560 8.6 and 7.5 us, 512 x 4096 8.3 and 7.6, 4096 x 4096 12.1 and 10.8, q, k, v of an 8B layer 12.9 and 12.8; above
// the line one layer of the 8B model 33.4 and 36.1).
static cudaError_t make_plan(const Problem* problems, int matrices, int sms, size_t ws_bytes, unsigned char** plan, size_t* meta_bytes) {
    long long exact_cols = 0, tasks = 0;
    int count = 0;  // of slices
    for (int i = 0; i < matrices; ++i) {
        exact_cols += problem_blocks(problems[i]);
        tasks += (long long)((problems[i].N + 7) / 8) * ((problem_blocks(problems[i]) + 31) / 32);
        count += problem_slices(problems[i]);
    }
    const int max_ranges = sms * kUnitWarps;
    const size_t all = plan_meta_bytes(count, max_ranges, 4 * count);
    unsigned char* buf = static_cast<unsigned char*>(calloc(1, all + size_t(count) * sizeof(MatrixUnits)));
    if (!buf) return cudaErrorMemoryAllocation;
    PlanHeader* H = reinterpret_cast<PlanHeader*>(buf);
    H->count = count;
    // Matrices whose units are longest come first, so that the units claimed at the end are short (14B, 6 / 16 / 36 layers
    // 260 / 637 / 1394 -> 242 / 620 / 1375 us).  What a row's sum is made of does not depend on the order, but where a unit is
    // cut does, and with it the order of its sums: the same plan gives the same bits, another list or order may differ in the last.
    Problem* problems_host = reinterpret_cast<Problem*>(buf + sizeof(PlanHeader));
    auto longest = [](const Problem& q) {
        const int Bi = problem_blocks(q);
        return groups_per_unit(Bi, kMaxRowGroups) * (Bi / 32) + (Bi % 32 ? 1 : 0);
    };
    for (int i = 0, at = 0; i < matrices; ++i)
        for (int k = 0, n = problem_slices(problems[i]); k < n; ++k) problems_host[at++] = n == 1 ? problems[i] : problem_slice(problems[i], k);
    auto before = [&](const Problem& a, const Problem& b) { return longest(a) > longest(b); };
    if (!std::is_sorted(problems_host, problems_host + count, before)) std::stable_sort(problems_host, problems_host + count, before);
    H->off_problems = uint32_t(sizeof(PlanHeader));
    H->off_unit_prefix = H->off_problems + uint32_t(count) * uint32_t(sizeof(Problem));
    H->off_col_prefix = H->off_unit_prefix + uint32_t(count + 1) * 4u;
    H->off_cuts = H->off_col_prefix + uint32_t(count + 1) * 4u;
    int32_t* up = reinterpret_cast<int32_t*>(buf + H->off_unit_prefix);
    int32_t* cp = reinterpret_cast<int32_t*>(buf + H->off_col_prefix);
    if (exact_cols + 31LL * count > 0x7FFFFFF0LL) { free(buf); return cudaErrorInvalidValue; }
    MatrixUnits* M = reinterpret_cast<MatrixUnits*>(buf + all);
    auto place_units = [&](int row_groups) {
        long long units = 0;
        for (int i = 0; i < count; ++i) {
            const int B = problem_blocks(problems_host[i]), R = groups_per_unit(B, row_groups), G = (problems_host[i].N + 7) / 8;
            M[i] = MatrixUnits{R, G, B / 32, B % 32 > 0, (G + R - 1) / R};
            up[i] = int32_t(units);
            units += M[i].units;
        }
        up[count] = H->total_units = int32_t(units);
        H->row_groups = row_groups;
        return units <= 0x7FFFFFF0LL;
    };
    auto place_columns = [&](bool aligned) {
        long long cols = 0;
        for (int i = 0; i < count; ++i) {
            cp[i] = int32_t(cols);
            if (i + 1 == count || !same_columns(problems_host[i], problems_host[i + 1])) cols += problem_cols(problems_host[i], aligned);
        }
        cp[count] = H->total_cols = int32_t(cols);
        H->aligned = aligned;
    };
    size_t meta = 0, slots = 0;
    auto fits = [&](bool aligned) {  // and where everything lies
        place_columns(aligned);
        const int ranges = H->warps_per_cta * sms;
        H->off_col_start = H->off_cuts + uint32_t(ranges ? (ranges + 1) * sizeof(WarpCut) : 0);
        H->col_shift = col_shift_for(size_t(H->total_cols), count);
        meta = plan_meta_bytes(count, ranges, (H->total_cols >> H->col_shift) + 1);
        const size_t bytes = plan_bytes(meta, H->counters, slots, size_t(H->total_cols));
        H->off_counters = uint32_t(meta);
        H->off_partials = H->off_counters + uint32_t(H->counters) * 4u;
        H->off_xq = uint32_t(bytes - size_t(H->total_cols) * kXqBytesPerCol);
        return bytes <= ws_bytes;
    };
    WarpCut* cuts = reinterpret_cast<WarpCut*>(buf + H->off_cuts);
    bool room = false;
    for (int way = tasks <= 2LL * max_ranges ? 1 : 0; way < 4 && !room; ++way) {
        const bool inside = way < 2;
        if (!place_units(way == 1 ? 1 : kMaxRowGroups)) break;
        H->nwarps = way < 3 ? max_ranges : 0;
        if (way < 3) {
            slots = cut_ranges(H, M, up, cuts, sms, inside);
        } else {
            H->warps_per_cta = H->counters = 0;
            slots = 0;
            H->dyn_start = H->total_units;
        }
        room = slots <= 65536 && (fits(true) || fits(false));
    }
    if (!room) { free(buf); return cudaErrorInvalidValue; }
    int32_t* start = reinterpret_cast<int32_t*>(buf + H->off_col_start);
    for (int c = 0, i = 0; c <= H->total_cols >> H->col_shift; ++c) {
        while (i < count - 1 && cp[i + 1] <= (long long)c << H->col_shift) ++i;
        start[c] = i;
    }
    *plan = buf;
    *meta_bytes = meta;
    return cudaSuccess;
}

cudaError_t grouped_plan(const Problem* problems, int matrices, void* ws_dev, size_t ws_bytes, cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    unsigned char* plan = nullptr;
    size_t meta = 0;
    e = make_plan(problems, matrices, sms, ws_bytes, &plan, &meta);
    if (e != cudaSuccess) return e;
    // pageable source: the runtime stages it before returning, so the buffer can be freed
    e = cudaMemcpyAsync(ws_dev, plan, meta, cudaMemcpyHostToDevice, s);
    free(plan);
    return e;
}

size_t single_plan_meta_bytes() { return plan_meta_bytes(1, 0, 1); }

size_t single_plan_scratch_bytes(int blocks_per_row) {
    return single_plan_meta_bytes() + size_t((blocks_per_row + 31) & ~31) * kXqBytesPerCol;
}

void single_plan_fill(const Problem& problem, unsigned char* meta_host) {
    memset(meta_host, 0, single_plan_meta_bytes());
    PlanHeader* H = reinterpret_cast<PlanHeader*>(meta_host);
    H->count = 1;
    H->row_groups = kMaxRowGroups;
    H->aligned = 1;
    H->total_units = problem_units(problem, kMaxRowGroups);
    H->total_cols = int32_t(problem_cols(problem, true));
    H->off_problems = uint32_t(sizeof(PlanHeader));
    H->nwarps = 0;  // no unit ranges: the kernel deals units round-robin
    H->off_unit_prefix = H->off_problems + uint32_t(sizeof(Problem));
    H->off_col_prefix = H->off_unit_prefix + 8u;
    H->off_xq = uint32_t(single_plan_meta_bytes());
    memcpy(meta_host + H->off_problems, &problem, sizeof(Problem));
    int32_t* up = reinterpret_cast<int32_t*>(meta_host + H->off_unit_prefix);
    int32_t* cp = reinterpret_cast<int32_t*>(meta_host + H->off_col_prefix);
    up[0] = 0; up[1] = H->total_units;
    cp[0] = 0; cp[1] = H->total_cols;
    H->off_col_start = H->off_col_prefix + 8u;  // one entry, zero: one matrix
    H->col_shift = 31;
    H->dyn_start = H->total_units;
}

cudaError_t grouped_run(void* ws_dev, const void* table, cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const uint32_t smem = kTableSmemBytes + kUnitWarps * kUnitFloats * 4 + kUnitWarps * 3072;
    static PerDeviceOnce once;
    e = once.run([smem] { return cudaFuncSetAttribute(k_gemv_units, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)); });
    if (e != cudaSuccess) return e;
    e = launch_pdl(k_prepare_x, sms * 4, 128, 0, s, static_cast<unsigned char*>(ws_dev));
    if (e != cudaSuccess) return e;
    return launch_pdl(k_gemv_units, sms, kUnitThreads, smem, s, static_cast<const DeviceTables*>(table),
                      static_cast<unsigned char*>(ws_dev));
}

}  // namespace tetra
