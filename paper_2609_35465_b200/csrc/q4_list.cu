// Batch-1 products of a LIST of 4-bit group-quantised matrices (the int4 projections of a token pass,
// Sec. 4.1, 4.3, 5.1) from one persistent grid.
//
// A single tetra_q4_gemv launch on a projection-sized matrix (2-27 MB) is over in a few microseconds,
// most of them fixed cost: the launch, the per-CTA prologue (group sums of the activations behind a
// barrier), the ring filling up, the pieces combined behind another barrier.  Here the chunks of all
// matrices form one sequence in memory order; every warp of a persistent grid owns a contiguous
// range of it and streams it through its cp.async ring without ever draining it between matrices,
// and no warp waits for another.  One kernel:
//   * per group of the activations the sum of x and minus the sum of bias_k x_k (the MMA operands carry biases
//     1024 and 64) are made by each CTA for the few matrices its warps meet, in shared memory, while the first
//     chunks are on their way, and the activations stay in shared memory with them.  (Read through L1 they queue behind
//     the chunks' copies, which the same unit takes in order: a warp then waits for its newest copy before it can
//     multiply its oldest chunk, and more copies in flight make it worse.  36 layers, 1.37 GB: 269 us from idle and
//     284 us under the board's power limit; with the activations in shared memory 201 us from idle and, by the board,
//     227 to 244 us under the limit);
//   * the stream: dequantise with five logic operations per four registers, MMA against the activations, scale
//     and offset per group; a strip (32 rows) that lies wholly inside a warp's range is stored; one cut by range
//     boundaries leaves a piece per warp in the workspace, and the warp that finds the strip's other pieces there
//     adds them in warp order and stores it.
// Where a warp starts and who shares its strips is written into the plan: searched for on the device it was a chain
// of dependent loads in every warp.  (One layer's projections, 38 MB: 22.5 us with searches, a kernel before this one
// for the group sums and one after it for the pieces; now 12.5 us.)
// Deterministic (fixed order everywhere); nothing waits for another warp (a counter per cut strip only tells the
// last one); CTA barriers, cp.async.wait_group and griddepcontrol.wait are the only waits.
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "../../include/tetra.h"
#include "../../include/tetra_q4.h"
#include "q4_common.cuh"
#include "tetra_gemv_common.cuh"

namespace tetra {
namespace {

constexpr int kQ4ListThreads = 512;
constexpr int kQ4ListWarps = kQ4ListThreads / 32;
constexpr int kPieceFloats = 32;  // a partial strip: column 0 of its 32 rows (the list call has one vector per matrix)

struct Q4Item {
    const unsigned char* packed;
    const __half* x;
    float* y;
    int32_t N;
    int32_t groups, strips;
    uint32_t chunk_begin;  // chunks of the matrices before this one
    uint32_t group_begin;  // groups of the matrices before this one (index into the group sums)
    uint32_t pad_;
};
static_assert(sizeof(Q4Item) == 48, "descriptor layout");

// What a warp's range [c_begin, c_end) of the chunk sequence meets, known when the list is planned.
struct Q4Warp {
    int32_t item;    // matrix of its first chunk
    int32_t owner;   // warp in whose range the strip of its first chunk begins
    int32_t parts;   // pieces of the strip that begins in this range and ends beyond it (0: there is none)
    int32_t arrived; // of those pieces, how many are there (zero between runs)
};

struct Q4ListHeader {
    int32_t nwarps;
    uint32_t total_chunks;
    uint32_t off_items, off_warps, off_pieces;
};

inline size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

struct Q4ListLayout {
    size_t off_items, off_warps, off_pieces, total;
};
Q4ListLayout list_layout(int count, int nwarps) {
    Q4ListLayout L;
    L.off_items = align256(sizeof(Q4ListHeader));
    L.off_warps = align256(L.off_items + size_t(count) * sizeof(Q4Item));
    L.off_pieces = align256(L.off_warps + size_t(nwarps) * sizeof(Q4Warp));
    L.total = align256(L.off_pieces + size_t(nwarps) * 2 * kPieceFloats * 4);
    return L;
}

// First chunk of warp w's range.
__host__ __device__ inline uint32_t range_begin(uint32_t total, int w, int nw) { return uint32_t(uint64_t(total) * uint32_t(w) / uint32_t(nw)); }

// Bytes of activations that a CTA holds in shared memory, beside the rings: five vectors of 8192.  A CTA whose warps meet
// more (short matrices: their activations outweigh their rows) reads them through L1 and makes the sums chunk by chunk.
constexpr uint32_t kQ4ListX = 80 * 1024;
template <int G>
__host__ __device__ constexpr uint32_t list_held_groups() { return kQ4ListX / (2 * G); }

// (sum x, minus the sum of bias_k x_k) of one group, bias 1024 for k % 4 in {0, 1} and 64 for {2, 3}; LANES consecutive
// lanes each hold every LANES-th four activations (and copy them to `keep`), all of them get the result.
template <int G, int LANES, bool KEEP>
__device__ __forceinline__ float2 group_sums(const __half* x, int sub, uint2* keep) {
    const uint2* src = reinterpret_cast<const uint2*>(x);
    float lo = 0.f, hi = 0.f;
#pragma unroll
    for (int i = 0; i < G / 4; i += LANES) {
        const uint2 u = G / 4 >= LANES || sub < G / 4 ? __ldg(src + sub + i) : make_uint2(0u, 0u);
        if (KEEP) keep[sub + i] = u;
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        lo += a.x + a.y;
        hi += b.x + b.y;
    }
#pragma unroll
    for (int o = LANES / 2; o >= 1; o >>= 1) {
        lo += __shfl_xor_sync(0xFFFFFFFFu, lo, o);
        hi += __shfl_xor_sync(0xFFFFFFFFu, hi, o);
    }
    return make_float2(lo + hi, -(1024.f * lo + 64.f * hi));
}

template <int G, int DEPTH>
__global__ void __launch_bounds__(kQ4ListThreads, 1) k_q4_list_main(unsigned char* __restrict__ ws) {
    constexpr int TPG = G / 64, CH = q4_chunk_bytes(G), PIECES = CH / 16;
    extern __shared__ __align__(16) unsigned char q4_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    pdl_release();
    // the plan (written once, long before) and the weights do not depend on the preceding kernel
    const Q4ListHeader* H = reinterpret_cast<const Q4ListHeader*>(ws);
    const Q4Item* items = reinterpret_cast<const Q4Item*>(ws + H->off_items);
    // behind the rings: the held groups' sums, zeros for the B columns without a vector, the held groups' activations
    float2* sums = reinterpret_cast<float2*>(q4_smem + size_t(kQ4ListWarps) * DEPTH * CH);
    unsigned char* zeros = reinterpret_cast<unsigned char*>(sums + list_held_groups<G>());
    unsigned char* held_x = zeros + kQ4TileZeros;
    float* pieces = reinterpret_cast<float*>(ws + H->off_pieces);
    Q4Warp* warps = reinterpret_cast<Q4Warp*>(ws + H->off_warps);
    // A list of fewer chunks than warps uses as many warps as chunks, spread over the CTAs.
    const int nw = H->nwarps, all = int(gridDim.x) * kQ4ListWarps;
    const int gw = nw < all ? warp * int(gridDim.x) + int(blockIdx.x) : int(blockIdx.x) * kQ4ListWarps + warp;
    const bool work = gw < nw;
    const uint32_t total = H->total_chunks;
    const uint32_t c_begin = work ? range_begin(total, gw, nw) : 0u, c_end = work ? range_begin(total, gw + 1, nw) : 0u;
    const int first_item = work ? warps[gw].item : 0;

    const uint32_t ring_lane = smem_u32(q4_smem) + uint32_t(warp) * (DEPTH * CH) + lane * 16;
    const uint32_t ring_lane_end = ring_lane + DEPTH * CH;
    const bool tail_lane = lane < PIECES % 32;  // lanes that copy the last, partial group of 16-byte pieces

    // fetch side: the next chunk to copy, wherever in the list it lies
    int fi = first_item;
    uint32_t f_left_in_item = items[fi].chunk_begin + uint32_t(items[fi].groups) * uint32_t(items[fi].strips) - c_begin;
    const unsigned char* f_src = items[fi].packed + size_t(c_begin - items[fi].chunk_begin) * CH + lane * 16;
    int f_todo = int(c_end - c_begin);
    auto fetch_into = [&](uint32_t dst_lane) {
        if (f_todo > 0) {
#pragma unroll
            for (int i = 0; i < PIECES / 32; ++i) q4_cp_async16(dst_lane + i * 512, f_src + i * 512);
            if (PIECES % 32 != 0 && tail_lane) q4_cp_async16(dst_lane + (PIECES / 32) * 512, f_src + (PIECES / 32) * 512);
            f_src += CH;
            if (--f_left_in_item == 0 && f_todo > 1) {  // on to the next matrix of the list
                ++fi;
                f_src = items[fi].packed + lane * 16;
                f_left_in_item = uint32_t(items[fi].groups) * uint32_t(items[fi].strips);
            }
        }
        --f_todo;
        asm volatile("cp.async.commit_group;" ::: "memory");  // one group per call, empty or not
    };
#pragma unroll
    for (int i = 0; i < DEPTH - 1; ++i) fetch_into(ring_lane + i * CH);

    // the matrices of this CTA's warps follow one another, and so do their groups
    const int cta_first = int(blockIdx.x) * kQ4ListWarps, cta_next = min(cta_first + kQ4ListWarps, nw - 1);
    const bool spread = nw < all;
    const int item_lo = spread ? 0 : warps[cta_first].item, item_hi = spread ? 0 : warps[cta_next].item;
    const uint32_t group_lo = items[item_lo].group_begin;
    const bool held = !spread && items[item_hi].group_begin + uint32_t(items[item_hi].groups) - group_lo <= list_held_groups<G>();
    pdl_wait();  // the activations may come from a kernel before
    if (held) {
        for (int it = item_lo; it <= item_hi; ++it) {
            const Q4Item I = items[it];
            // eight lanes per group; the whole warp goes round, so that all lanes are there for the shuffles
            for (int k0 = warp * 4; k0 < I.groups; k0 += kQ4ListWarps * 4) {
                const int k = min(k0 + (lane >> 3), I.groups - 1);
                const uint32_t at = I.group_begin - group_lo + uint32_t(k);
                const float2 v = group_sums<G, 8, true>(I.x + size_t(k) * G, lane & 7, reinterpret_cast<uint2*>(held_x + size_t(at) * (2 * G)));
                if ((lane & 7) == 0) sums[at] = v;
            }
        }
        if (threadIdx.x < kQ4TileZeros / 16) reinterpret_cast<uint4*>(zeros)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    }
    if (!work) return;

    uint32_t slot_lane = ring_lane;                       // slot being consumed
    uint32_t refill_lane = ring_lane + (DEPTH - 1) * CH;  // slot consumed last (empty at the start)
    const uint32_t so_delta = uint32_t(TPG * 1024 + g * 4) - uint32_t(lane * 16);  // slot_lane -> this lane's scale records

    // consume side
    int ci = first_item;
    uint32_t left = c_end - c_begin;
    uint32_t local = c_begin - items[ci].chunk_begin;  // chunk index inside matrix ci
    auto stream = [&](auto in_shared) {
        constexpr bool HELD = decltype(in_shared)::value;
        while (left > 0) {
            const Q4Item I = items[ci];
            const int groups = I.groups;
            int strip = int(local / uint32_t(groups));
            int gi = int(local - uint32_t(strip) * uint32_t(groups));
            uint32_t in_item = min(left, uint32_t(groups) * uint32_t(I.strips) - local);
            left -= in_item;
            local += in_item;
            // Column 0 of the B fragment is the activation vector.  The other columns are never stored and read zeros wherever
            // the walk is: multiplying zeros takes less power, and long lists run at the board's limit.
            const auto x_lane = [&] {
                if constexpr (HELD) return g == 0 ? smem_u32(held_x) + (I.group_begin - group_lo) * (2u * G) + 32u * t : smem_u32(zeros);
                else return reinterpret_cast<const unsigned char*>(g == 0 ? reinterpret_cast<const uint4*>(I.x + 16 * t) : q4_zeros);
            }();
            const uint32_t x_step = g == 0 ? 2u * G : 0u;
            const float2* item_sums = sums + (I.group_begin - group_lo);
            while (in_item > 0) {
                // one segment: the chunks of this warp that belong to one strip
                const int seg_first = gi;
                const uint32_t seg_len = min(uint32_t(groups - gi), in_item);
                auto xp = x_lane + uint32_t(gi) * x_step;
                float acc[2][2] = {};  // column 2 t of rows 16 h + g, 16 h + g + 8
                for (uint32_t c = 0; c < seg_len; ++c, ++gi) {
                    const float2 cs = HELD ? item_sums[gi] : group_sums<G, 32, false>(I.x + size_t(gi) * G, lane, nullptr);
                    [[maybe_unused]] uint32_t xl[TPG][8];
                    if constexpr (!HELD) load_group<TPG>(xp, xl);  // ahead of the copies: see there
                    fetch_into(refill_lane);
                    q4_cp_async_wait<DEPTH - 1>();  // this chunk has landed
                    __syncwarp();
                    float d[2][4];
#pragma unroll
                    for (int j = 0; j < TPG; ++j) {
                        uint32_t xr[8];
                        if constexpr (HELD) {
                            uint32_t lo[4], hi[4];
                            q4_lds128(xp + 128 * j, lo);
                            q4_lds128(xp + 128 * j + 16, hi);
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
                                    mma_f16_first(d[h], a, xr[0], xr[1], cs.y, 0.f);
                                else
                                    mma_f16(d[h], a, xr[2 * m], xr[2 * m + 1]);
                            }
                        }
                    }
                    const uint32_t so_lane = slot_lane + so_delta;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t so0 = lds32(so_lane + 64 * h);
                        const uint32_t so1 = lds32(so_lane + 64 * h + 32);
                        const float2 r0 = __half22float2(*reinterpret_cast<const __half2*>(&so0));  // (scale, offset)
                        const float2 r1 = __half22float2(*reinterpret_cast<const __half2*>(&so1));
                        acc[h][0] = fmaf(r0.x, d[h][0], fmaf(r0.y, cs.x, acc[h][0]));
                        acc[h][1] = fmaf(r1.x, d[h][2], fmaf(r1.y, cs.x, acc[h][1]));
                    }
                    xp += x_step;
                    __syncwarp();  // every lane has read the slot before the next refill targets it
                    refill_lane = slot_lane;
                    slot_lane += CH;
                    if (slot_lane == ring_lane_end) slot_lane = ring_lane;
                }
                in_item -= seg_len;
                if (seg_first == 0 && gi == groups) {  // the whole strip was this warp's: store column 0
                    if (t == 0) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int row = 32 * strip + 16 * h + g + 8 * i;
                                if (row < I.N) I.y[row] = acc[h][i];
                            }
                    }
                } else {
                    // A strip shared with neighbouring warps: leave a piece (column 0: floats 4 g .. 4 g + 3 = rows g, g + 8,
                    // 16 + g, 24 + g).  A warp has at most one strip that began before its range (slot 0) and one that ends
                    // beyond it (slot 1).
                    const bool later = seg_first != 0;  // began before this range
                    if (t == 0)
                        *reinterpret_cast<float4*>(pieces + (size_t(2 * gw) + (later ? 0 : 1)) * kPieceFloats + 4 * g) =
                            make_float4(acc[0][0], acc[0][1], acc[1][0], acc[1][1]);
                    const int owner = later ? warps[gw].owner : gw, parts = warps[owner].parts;
                    __threadfence();  // the piece is visible before the counter moves
                    __syncwarp();
                    int arrived = 0;
                    if (lane == 0) arrived = atomicAdd(&warps[owner].arrived, 1);
                    arrived = __shfl_sync(0xFFFFFFFFu, arrived, 0);
                    if (arrived == parts - 1) {  // all pieces are there: add them in warp order
                        __threadfence();
                        float sum = __ldcg(pieces + (size_t(2 * owner) + 1) * kPieceFloats + lane);
                        for (int k = 1; k < parts; ++k) sum += __ldcg(pieces + size_t(2 * (owner + k)) * kPieceFloats + lane);
                        const int row = 32 * strip + (lane >> 2) + 8 * (lane & 1) + 16 * ((lane >> 1) & 1);
                        if (row < I.N) I.y[row] = sum;
                        if (lane == 0) warps[owner].arrived = 0;  // for the next run
                    }
                }
                if (gi == groups) {
                    gi = 0;
                    ++strip;
                }
            }
            ++ci;
            local = 0;
        }
    };
    if (held) stream(std::true_type{});
    else stream(std::false_type{});
    q4_cp_async_wait<0>();
}

int check_list(const tetra_q4_problem* p, int count, int G) {
    if (!p) return TETRA_ERR_NULL;
    if (count <= 0 || count > TETRA_Q4_LIST_MAX) return TETRA_ERR_SHAPE;
    if (G != 64 && G != 128) return TETRA_ERR_SHAPE;
    for (int i = 0; i < count; ++i) {
        if (!p[i].packed || !p[i].x || !p[i].y) return TETRA_ERR_NULL;
        if (p[i].N <= 0 || p[i].K <= 0 || p[i].K > TETRA_Q4_MAX_K || p[i].K % G) return TETRA_ERR_SHAPE;
        if ((reinterpret_cast<uintptr_t>(p[i].packed) & 15) || (reinterpret_cast<uintptr_t>(p[i].x) & 15) ||
            (reinterpret_cast<uintptr_t>(p[i].y) & 3))
            return TETRA_ERR_ALIGN;
    }
    return TETRA_OK;
}

template <int G, int DEPTH>
cudaError_t run_main(unsigned char* ws, int sms, cudaStream_t s) {
    const size_t smem = size_t(kQ4ListWarps) * DEPTH * q4_chunk_bytes(G) + list_held_groups<G>() * sizeof(float2) + kQ4TileZeros + kQ4ListX;
    static PerDeviceOnce once;
    cudaError_t e = once.run([smem] {
        return cudaFuncSetAttribute(k_q4_list_main<G, DEPTH>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    });
    if (e != cudaSuccess) return e;
    return launch_pdl(k_q4_list_main<G, DEPTH>, sms, kQ4ListThreads, smem, s, ws);
}

}  // namespace
}  // namespace tetra

using namespace tetra;

extern "C" {

size_t tetra_q4_list_workspace_bytes(const tetra_q4_problem* problems_host, int count, int G) {
    if (check_list(problems_host, count, G) != TETRA_OK) return 0;
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return 0;
    return list_layout(count, sms * kQ4ListWarps).total;
}

int tetra_q4_list_plan(const tetra_q4_problem* problems_host, int count, int G, void* workspace_dev,
                       size_t workspace_bytes, void* stream) {
    const int rc = check_list(problems_host, count, G);
    if (rc != TETRA_OK) return rc;
    if (!workspace_dev) return TETRA_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return TETRA_ERR_ALIGN;
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return TETRA_ERR_CUDA;
    const int nwarps = sms * kQ4ListWarps;
    uint64_t chunks = 0;
    for (int i = 0; i < count; ++i) {
        const uint64_t gr = uint64_t(problems_host[i].K / G), st = uint64_t((problems_host[i].N + 31) / 32);
        chunks += gr * st;
    }
    if (chunks > 0x7FFFFFF0ull) return TETRA_ERR_SHAPE;  // strips and groups are no more than chunks
    const Q4ListLayout L = list_layout(count, nwarps);
    if (workspace_bytes < L.total) return TETRA_ERR_SIZE;
    const size_t meta = L.off_pieces;
    unsigned char* buf = static_cast<unsigned char*>(std::calloc(1, meta));
    if (!buf) return TETRA_ERR_CUDA;
    Q4ListHeader* H = reinterpret_cast<Q4ListHeader*>(buf);
    const int ranges = chunks < uint64_t(nwarps) ? int(chunks) : nwarps;  // no range is empty
    H->nwarps = ranges;
    H->total_chunks = uint32_t(chunks);
    H->off_items = uint32_t(L.off_items);
    H->off_warps = uint32_t(L.off_warps);
    H->off_pieces = uint32_t(L.off_pieces);
    Q4Item* items = reinterpret_cast<Q4Item*>(buf + L.off_items);
    uint32_t cb = 0, gb = 0;
    for (int i = 0; i < count; ++i) {
        const tetra_q4_problem& q = problems_host[i];
        Q4Item& I = items[i];
        I.packed = static_cast<const unsigned char*>(q.packed);
        I.x = static_cast<const __half*>(q.x);
        I.y = q.y;
        I.N = q.N;
        I.groups = q.K / G;
        I.strips = (q.N + 31) / 32;
        I.chunk_begin = cb;
        I.group_begin = gb;
        cb += uint32_t(I.groups) * uint32_t(I.strips);
        gb += uint32_t(I.groups);
    }
    Q4Warp* warps = reinterpret_cast<Q4Warp*>(buf + L.off_warps);
    int item = 0, owner = 0;
    uint32_t strip_at = 0xFFFFFFFFu;  // first chunk of the strip that the ranges so far have left open
    for (int w = 0; w < ranges; ++w) {
        const uint32_t begin = range_begin(uint32_t(chunks), w, ranges), end = range_begin(uint32_t(chunks), w + 1, ranges);
        auto strip_of = [&](uint32_t c) {  // first chunk of c's strip, c in matrix `item`
            const Q4Item& I = items[item];
            return I.chunk_begin + (c - I.chunk_begin) / uint32_t(I.groups) * uint32_t(I.groups);
        };
        auto advance = [&](uint32_t c) {
            while (item + 1 < count && items[item + 1].chunk_begin <= c) ++item;
        };
        advance(begin);
        warps[w].item = item;
        if (strip_of(begin) == strip_at) {  // shared with earlier ranges
            warps[w].owner = owner;
            ++warps[owner].parts;
        } else {
            warps[w].owner = w;
        }
        advance(end - 1);
        const uint32_t last = strip_of(end - 1);
        const bool open = end < last + uint32_t(items[item].groups);  // goes on in the next range
        if (!open) strip_at = 0xFFFFFFFFu;
        else if (last != strip_at) {
            strip_at = last;
            owner = w;
            warps[w].parts = 1;
        }
    }
    // pageable source: the runtime has taken its copy when the call returns, so the buffer can be freed
    const cudaError_t e = cudaMemcpyAsync(workspace_dev, buf, meta, cudaMemcpyHostToDevice, static_cast<cudaStream_t>(stream));
    std::free(buf);
    return e == cudaSuccess ? TETRA_OK : TETRA_ERR_CUDA;
}

int tetra_q4_list_run(void* workspace_dev, int G, void* stream) {
    if (!workspace_dev) return TETRA_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return TETRA_ERR_ALIGN;
    if (G != 64 && G != 128) return TETRA_ERR_SHAPE;
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return TETRA_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char* ws = static_cast<unsigned char*>(workspace_dev);
    const cudaError_t e = G == 128 ? run_main<128, 3>(ws, sms, s) : run_main<64, 6>(ws, sms, s);
    return e == cudaSuccess ? TETRA_OK : TETRA_ERR_CUDA;
}

}  // extern "C"
