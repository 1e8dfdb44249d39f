// Decode-and-multiply (Eq. (2), Sec. 5.1) for ONE matrix or a short list of
// matrices in a single launch, with no scratch memory: the kernel behind
// tetra_gemv, tetra_gemv_tail and tetra_gemv_list.
//
// Sec. 5.2 of the paper times one launch per matrix; on B200 such a launch holds
// a few microseconds of work, so what is left of it is a chain of latencies:
// dependency wait, activations, their fixed-point image, the passes, the sums.
// The kernel is arranged to shorten that chain (q, k, v of an 8B layer: 6.8 us a
// launch.  %globaltimer stamps in an arrangement that took 8.5: 1.3 us of prologue
// instructions ahead of the wait, 1.3 us of image, 3.1 us of passes, 0.7 us of
// epilogue, and CTAs that straddled two matrices and finished 2.5 us after the others):
//   * one CTA of sixteen warps per SM: the image and the tables are built and
//     fetched once per SM (two CTAs of eight warps, which let the next launch start
//     in the gaps of this one, spend more on doing both twice: q, k, v 1.5 us more);
//   * a CTA works on ONE matrix; the host cuts every matrix's row groups into the
//     CTAs' shares, and the kernel finds its share with a few comparisons of
//     parameters: no division, no chain of loads;
//   * everything that does not depend on the activations is requested before the
//     wait for the predecessor in the stream (programmatic dependent launch) and
//     waited for only after the image has been built: the decode tables, every
//     warp's first code record, row scales, tails;
//   * the image takes a thread per (column, section), eight activations each, as
//     long as there is a thread for each, and beyond a thread per column;
//   * the warps split the CTA's passes evenly in memory order, a pass being 32
//     consecutive (row group, column) cells: where a row ends inside a pass the
//     next row group's first columns fill the lanes.  A row group is a record's
//     eight rows or (R = 4) half of them, whichever leaves the last pass of the
//     busiest warp earlier;
//   * per-(row group, warp) partial sums meet in shared memory and are added in
//     warp order (deterministic), then row scale and tail.
// The only waits are CTA barriers, cp.async.wait_group and griddepcontrol.wait.
#include "../../include/tetra.h"
#include "tetra_gemv_common.cuh"

namespace tetra {

static_assert(kListMax == TETRA_LIST_MAX, "list length limit must agree with the header");

constexpr int kListWarps = 16, kListThreads = 32 * kListWarps;
// A CTA's rows are taken in chunks whose partial sums, scales and tails share shared memory; a chunk has at least this
// many rows if the CTA has them, and more where there is room: see launch_gemv_list.
constexpr int kChunkRows = 128;

// Kernel parameters: the list and its split over the grid.  CTAs [cta_begin[i], cta_begin[i + 1]) work on matrix i
// (entries beyond the list: never reached); the first `extra` of them take base + 1 row groups, the others base.
// What a CTA needs of its matrix is one 64-byte line of constant memory: parameters are cold in every launch.
struct alignas(64) ListMatrix {
    const void* codes;
    const __half* x;
    const float* row_scales;
    const __half* tail;
    float* y;
    int32_t N, K;
    int32_t base, extra;
    uint32_t inv_bs;  // ceil(2^32 / max(words per row, 32)): cell -> row group by one high multiply
    int32_t begin;    // first CTA
};
static_assert(sizeof(ListMatrix) == 64, "one line");
struct ListParams {
    int32_t cta_begin[kListMax];
    int32_t image_cols;         // largest number of words per row, if the image fits
    int32_t batch;
    int32_t chunk;              // row groups of a chunk
    ListMatrix m[kListMax];
};

struct ListSmem {
    // offsets from the 16 KiB-aligned table copy; total includes the alignment slack
    uint32_t xq, xtail, ring, part, rs, tail, total;
};
__host__ __device__ inline ListSmem list_smem(int image_cols, int chunk_rows) {  // chunk_rows: a multiple of eight
    ListSmem S;
    S.xq = uint32_t(kFastBytes);
    S.xtail = S.xq + uint32_t(image_cols) * kXqBytesPerCol;               // float [24]: x beyond the last word
    S.ring = S.xtail + 96u;
    S.part = S.ring + kListWarps * 3072u;
    S.rs = S.part + uint32_t(chunk_rows * kListWarps * 4);                // float [chunk rows]: row scales
    S.tail = S.rs + uint32_t(chunk_rows * 4);                             // half [chunk rows][24]: tails
    S.total = S.tail + uint32_t(chunk_rows * 24 * 2) + kSmAlign;
    return S;
}

// Record of one lane in the ring: R = 8: the three 16-byte parts at +0, +512, +1024; R = 4: the half's four w0 words
// at +0, its two w1 words at +1024.
template <int R>
__device__ __forceinline__ void ring_fetch(uint32_t dst, const uint4* codes, uint32_t Bu, int group, uint32_t col) {
    if (R == 8) {
        const uint4* rec = codes + size_t(group) * 3 * Bu + col;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(rec));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + 512), "l"(rec + Bu));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + 1024), "l"(rec + 2 * Bu));
    } else {
        const uint4* rec = codes + size_t(group >> 1) * 3 * Bu + col;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(rec + ((group & 1) ? Bu : 0u)));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" :: "r"(dst + 1024), "l"(reinterpret_cast<const uint2*>(rec + 2 * Bu) + (group & 1)));
    }
}

// Sums v[r] over the 32 lanes for r < R through a warp-private buffer (R x kRedStride floats); the result for row
// lane / (32 / R) ends up in all 32 / R lanes of that row.
template <int R>
__device__ __forceinline__ float warp_row_sums(float* red, int lane, const float (&v)[R]) {
    constexpr int L = 32 / R;  // lanes per row, R values each
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) red[r * kRedStride + lane] = v[r];
    __syncwarp();
    const float4* src = reinterpret_cast<const float4*>(red + (lane / L) * kRedStride + R * (lane % L));
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < R / 4; ++k) {
        const float4 q = src[k];
        s += (q.x + q.y) + (q.z + q.w);
    }
#pragma unroll
    for (int o = 1; o < L; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

// R: rows of a row group (8: a record, 4: half of one);
// IMAGE: the CTA keeps the fixed-point image of the matrix's activations in shared memory (one 80-byte record per
// column); otherwise (more columns than fit) a lane builds its column's record from x for every pass.
template <int R, bool IMAGE>
__global__ void __launch_bounds__(kListThreads, 1)
k_gemv_list(const DeviceTables* __restrict__ tab, const __grid_constant__ ListParams L) {
    constexpr int THREADS = kListThreads, W = kListWarps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_release();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int CHUNK = L.chunk;
    const ListSmem S = list_smem(IMAGE ? L.image_cols : 0, (CHUNK * R + 7) & ~7);
    const uint32_t sm_raw = smem_u32(smem_raw);
    unsigned char* smem = smem_raw + (((sm_raw + kSmAlign - 1) & ~(kSmAlign - 1)) - sm_raw);
    const uint32_t sm_tab = smem_u32(smem);
    float* part = reinterpret_cast<float*>(smem + S.part);
    float* xtail = reinterpret_cast<float*>(smem + S.xtail);
    float* rs_sm = reinterpret_cast<float*>(smem + S.rs);
    __half* tail_sm = reinterpret_cast<__half*>(smem + S.tail);
    const uint32_t ring_base = S.ring + uint32_t(warp) * 3072u;
    const uint32_t ring = sm_tab + ring_base + uint32_t(lane) * 16u;

    // this CTA's matrix and row groups
    int p = 0;
#pragma unroll
    for (int i = 1; i < kListMax; ++i) p += int(blockIdx.x) >= L.cta_begin[i] ? 1 : 0;
    const ListMatrix& P = L.m[p];
    const int j = int(blockIdx.x) - P.begin;
    const int g_lo = j * P.base + min(j, P.extra);
    const int g_hi = g_lo + P.base + (j < P.extra ? 1 : 0);
    const uint32_t inv_bs = P.inv_bs;
    const int K = P.K, ntail = P.tail ? K % 24 : 0;
    const uint32_t Bu = uint32_t(P.tail ? K / 24 : (K + 23) / 24), Bs = Bu < 32u ? 32u : Bu;
    const uint4* codes = static_cast<const uint4*>(P.codes);

    // Geometry of a chunk (row groups [ga, ga + ng)): its cells (row group, column) are numbered row group by row
    // group, Bs to a row group (cells with column >= Bu are empty), a pass is 32 consecutive cells.
    auto fetch = [&](uint32_t dst, int ga, int ng, int rgl, uint32_t col) {
        ring_fetch<R>(dst, codes, Bu, ga + min(rgl, ng - 1), min(col, Bu - 1));
    };
    auto cell_of = [&](int ps, int& rgl, uint32_t& col) {
        const uint32_t cell = uint32_t(ps) * 32u + uint32_t(lane);
        const uint32_t r = __umulhi(cell, inv_bs);
        rgl = int(r);
        col = cell - r * Bs;
    };
    // Row scales and tails of a chunk's rows into shared memory; cp.async where the addresses allow it, so that
    // nothing here waits for memory.  Eight threads per row.
    auto stage_rows = [&](int ga, int ng) {
        const int rows = min(ng * R, P.N - ga * R);
        const float* rs = P.row_scales + size_t(ga) * R;
        for (int t = threadIdx.x; t < rows; t += THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(smem_u32(rs_sm + t)), "l"(rs + t));
        if (ntail) {
            const __half* tl = P.tail + size_t(ga) * R * ntail;
            const bool pairs = (ntail & 1) == 0 && (reinterpret_cast<uintptr_t>(tl) & 3) == 0;
            for (int t = threadIdx.x >> 3; t < rows; t += THREADS / 8) {
                if (pairs) {
                    for (int k = 2 * (threadIdx.x & 7); k < ntail; k += 16)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;"
                                     :: "r"(smem_u32(tail_sm + t * 24 + k)), "l"(tl + size_t(t) * ntail + k));
                } else {
                    for (int k = threadIdx.x & 7; k < ntail; k += 8) tail_sm[t * 24 + k] = tl[size_t(t) * ntail + k];
                }
            }
        }
    };

    // ---- before the wait: requests that do not depend on the activations ----------------------
    {
        const int ng = min(g_hi - g_lo, CHUNK);
        const int passes = int((uint32_t(ng) * Bs + 31u) >> 5);
        const int ps0 = passes * warp / W, ps1 = passes * (warp + 1) / W;
        if (ps0 < ps1) {
            int rgl;
            uint32_t col;
            cell_of(ps0, rgl, col);
            fetch(ring, g_lo, ng, rgl, col);
        }
        stage_fast_tables_async(tab, smem_raw);
        stage_rows(g_lo, ng);
        asm volatile("cp.async.commit_group;");
    }
    pdl_wait();  // the activations may come from the previous kernel of the stream

    // Image task: (column, section) `id`, from the column's pairs w.
    auto image_task = [&](uint32_t id, const uint32_t (&w)[12]) {
        const uint32_t s = (id >= Bu ? 1u : 0u) + (id >= 2 * Bu ? 1u : 0u), c = id - s * Bu;
        float inv;
        const float step = column_step(w, inv);
        const uint32_t w0 = s == 0 ? w[0] : (s == 1 ? w[4] : w[8]), w1 = s == 0 ? w[1] : (s == 1 ? w[5] : w[9]);
        const uint32_t w2 = s == 0 ? w[2] : (s == 1 ? w[6] : w[10]), w3 = s == 0 ? w[3] : (s == 1 ? w[7] : w[11]);
        uint32_t hi[2], mid[2], lo[2];
        quantise_section(w0, w1, w2, w3, inv, hi, mid, lo);
        unsigned char* rec = smem + S.xq + c * kXqBytesPerCol;
        *reinterpret_cast<uint2*>(rec + 8 * s) = make_uint2(hi[0], hi[1]);
        *reinterpret_cast<uint2*>(rec + 24 + 8 * s) = make_uint2(mid[0], mid[1]);
        *reinterpret_cast<uint2*>(rec + 48 + 8 * s) = make_uint2(lo[0], lo[1]);
        if (s == 0) *reinterpret_cast<float*>(rec + 72) = step;
    };
    // The three sections of column c.  With more sections than threads a thread takes a column and the activations are read
    // in one round instead of two or three, each of which waits for memory (4096 x 12288 9.95 -> 9.49 us, 1024 x 6000
    // 4.41 -> 4.03, 5003 x 7001 9.07 -> 8.89).  Up to a section per thread the shorter chain is the better one (4096 x 4096, 170 columns: image 0.5 us).
    const bool by_column = 3 * Bu > uint32_t(THREADS);
    auto image_sections = [&](uint32_t c, const uint32_t (&w)[12]) {
        float inv;
        const float step = column_step(w, inv);
        unsigned char* rec = smem + S.xq + c * kXqBytesPerCol;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            uint32_t hi[2], mid[2], lo[2];
            quantise_section(w[4 * s], w[4 * s + 1], w[4 * s + 2], w[4 * s + 3], inv, hi, mid, lo);
            *reinterpret_cast<uint2*>(rec + 8 * s) = make_uint2(hi[0], hi[1]);
            *reinterpret_cast<uint2*>(rec + 24 + 8 * s) = make_uint2(mid[0], mid[1]);
            *reinterpret_cast<uint2*>(rec + 48 + 8 * s) = make_uint2(lo[0], lo[1]);
        }
        *reinterpret_cast<float*>(rec + 72) = step;
    };
    auto image_column = [&](uint32_t id) { return int(id - (id >= 2 * Bu ? 2 * Bu : (id >= Bu ? Bu : 0u))); };

    int parity = 0;
    bool first_chunk = true;
    for (int job = 0; job < L.batch; ++job) {  // activation vector `job`
        const __half* xj = P.x + size_t(job) * K;
        float* yj = P.y + size_t(job) * P.N;
        // the first round's activations are requested, then the rest of what a chunk needs, then the image is built
        uint32_t w[12];
        if (IMAGE && threadIdx.x < (by_column ? Bu : 3 * Bu)) load_column(xj, K, by_column ? int(threadIdx.x) : image_column(threadIdx.x), w);
        const float xt = int(threadIdx.x) < ntail ? __half2float(xj[24 * Bu + threadIdx.x]) : 0.f;
        if (job > 0) {
            __syncthreads();  // the vector before is done with the image and the buffers
        } else {
            for (int i = threadIdx.x; i < min(g_hi - g_lo, CHUNK) * W * R; i += THREADS) part[i] = 0.f;
        }
        if (IMAGE) {
            if (!by_column) {
                if (threadIdx.x < 3 * Bu) image_task(threadIdx.x, w);
            } else {
                for (uint32_t c = threadIdx.x; c < Bu; c += THREADS) {
                    if (c != threadIdx.x) load_column(xj, K, int(c), w);
                    image_sections(c, w);
                }
            }
        }
        if (threadIdx.x < 24) xtail[threadIdx.x] = xt;
        for (int g = g_lo; g < g_hi; g += CHUNK) {
            const int ng = min(g_hi - g, CHUNK);
            const int passes = int((uint32_t(ng) * Bs + 31u) >> 5);
            if (!first_chunk) {
                __syncthreads();  // the epilogue before has read its buffers
                for (int i = threadIdx.x; i < ng * W * R; i += THREADS) part[i] = 0.f;
                stage_rows(g, ng);
                asm volatile("cp.async.commit_group;");
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();  // tables, rows and image are in place, the partial sums are zero

            // ---- this warp's passes --------------------------------------------------------
            const int ps0 = passes * warp / W, ps1 = passes * (warp + 1) / W;
            if (ps0 < ps1) {
                int rgl;
                uint32_t col;
                cell_of(ps0, rgl, col);
                if (!first_chunk) {
                    fetch(ring + uint32_t(parity * 1536), g, ng, rgl, col);
                    asm volatile("cp.async.commit_group;");
                }
                int rg_acc = __shfl_sync(0xFFFFFFFFu, rgl, 0);  // row group the accumulators belong to
                float acc[R];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = 0.f;
                // folds the accumulators of row group rg_acc into this warp's slot of the partial sums, through the
                // ring slot of the pass at hand, which every lane has read
                auto flush = [&]() {
                    const float sum = warp_row_sums<R>(reinterpret_cast<float*>(smem + ring_base + parity * 1536), lane, acc);
                    constexpr int PL = 32 / R;
                    if (lane % PL == 0) part[(rg_acc * W + warp) * R + lane / PL] = sum;
                    __syncwarp();  // the buffer has been read before the slot is filled again
                };
                for (int ps = ps0; ps < ps1; ++ps) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    const uint32_t src = ring + uint32_t(parity * 1536);
                    uint4 a, b, h;
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w) : "r"(src));
                    if (R == 8) {
                        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "r"(src + 512));
                        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(h.x), "=r"(h.y), "=r"(h.z), "=r"(h.w) : "r"(src + 1024));
                    } else {
                        asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(h.x), "=r"(h.y) : "r"(src + 1024));
                    }
                    // this lane's cell of the next pass: 32 cells on, at most one row group further
                    int nrgl = rgl;
                    uint32_t ncol = col + 32u;
                    if (ncol >= Bs) { ncol -= Bs; ++nrgl; }
                    if (ps + 1 < ps1) fetch(ring + uint32_t((parity ^ 1) * 1536), g, ng, nrgl, ncol);
                    asm volatile("cp.async.commit_group;");
                    const bool active = rgl < ng && col < Bu;
                    LaneX X;
                    {
                        uint32_t q[20];
                        if (IMAGE) {
                            const uint4* rec = reinterpret_cast<const uint4*>(smem + S.xq + min(col, Bu - 1) * kXqBytesPerCol);
#pragma unroll
                            for (int k = 0; k < 5; ++k) {
                                const uint4 u = rec[k];
                                q[4 * k] = u.x; q[4 * k + 1] = u.y; q[4 * k + 2] = u.z; q[4 * k + 3] = u.w;
                            }
                        } else {
                            quantise_column(xj, K, int(min(col, Bu - 1)), q);
                        }
                        lane_x_from_words(q, active, X);
                    }
                    // Lanes of the pass sit in row group rg_acc or, behind a row boundary, in the next one.
                    // The former add to the accumulators; the latter wait until the accumulators have been
                    // folded and then start the next row group's.
                    const int rg_last = __shfl_sync(0xFFFFFFFFu, rgl, 31);
                    if (rg_last == rg_acc) {
                        record_accumulate<R>(sm_tab, a, b, h, X, acc);
                    } else {
                        float v[R];
                        record_values<R>(sm_tab, a, b, h, X, v);
                        const bool mine = rgl == rg_acc;
#pragma unroll
                        for (int r = 0; r < R; ++r) acc[r] += mine ? v[r] : 0.f;
                        flush();
                        rg_acc = rg_last;
#pragma unroll
                        for (int r = 0; r < R; ++r) acc[r] = mine ? 0.f : v[r];
                    }
                    if (ps + 1 == ps1 && rg_acc < ng) flush();
                    parity ^= 1;
                    rgl = nrgl;
                    col = ncol;
                }
            }
            first_chunk = false;
            __syncthreads();
            // ---- epilogue: eight threads per row.  Thread k of a row takes the partial sums of slots k and k + 8
            // and every eighth tail product; three shuffles add them in a fixed order; row scale, tail (Sec. 5.1).
            for (int i = threadIdx.x; i < ng * R * 8; i += THREADS) {
                const int t = i >> 3, k8 = i & 7;
                const float* pr = part + (t / R) * W * R + t % R;
                float v = pr[R * k8] + pr[R * (k8 + 8)];
                v *= rs_sm[t];
                for (int k = k8; k < ntail; k += 8) v = fmaf(__half2float(tail_sm[t * 24 + k]), xtail[k], v);
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
                v += __shfl_xor_sync(0xFFFFFFFFu, v, 4);
                const int row = g * R + t;
                if (k8 == 0 && row < P.N) yj[row] = v;
            }
        }
    }
}

namespace {

struct ListShape {
    int rows[kListMax], blocks[kListMax];
    int count, max_blocks;
};

// Splits the list's row groups of R rows over at most `ctas` CTAs; fills P's shares and returns the CTAs used and
// the passes of the busiest warp and the row groups of the largest share.
int split_list(const ListShape& Q, int R, int ctas, ListParams& P, int* warp_passes, int* cta_groups) {
    int n[kListMax] = {}, groups[kListMax] = {}, used = 0;
    long long work = 0, total = 0;
    for (int i = 0; i < Q.count; ++i) {
        groups[i] = (Q.rows[i] + R - 1) / R;
        work += (long long)groups[i] * Q.blocks[i];
        total += groups[i];
    }
    if (total < ctas) ctas = int(total);
    auto cost = [&](int i, int c) { return (long long)((groups[i] + c - 1) / c) * Q.blocks[i]; };  // of a share, with c CTAs
    for (int i = 0; i < Q.count; ++i) {
        const long long share = (long long)groups[i] * Q.blocks[i] * ctas / work;
        n[i] = int(share < 1 ? 1 : (share > groups[i] ? groups[i] : share));
        used += n[i];
    }
    while (used < ctas) {  // what rounding left goes to the matrix whose CTAs are loaded most
        int at = -1;
        for (int i = 0; i < Q.count; ++i)
            if (n[i] < groups[i] && (at < 0 || cost(i, n[i]) > cost(at, n[at]))) at = i;
        if (at < 0) break;
        ++n[at];
        ++used;
    }
    while (used > ctas) {  // the smallest matrices took a whole CTA each
        int at = -1;
        for (int i = 0; i < Q.count; ++i)
            if (n[i] > 1 && (at < 0 || cost(i, n[i] - 1) < cost(at, n[at] - 1))) at = i;
        if (at < 0) break;
        --n[at];
        --used;
    }
    *warp_passes = *cta_groups = 0;
    int begin = 0;
    for (int i = 0; i < kListMax; ++i) {
        P.cta_begin[i] = i < Q.count ? begin : 0x7FFFFFFF;
        if (i >= Q.count) continue;
        ListMatrix& M = P.m[i];
        M.base = groups[i] / n[i];
        M.extra = groups[i] % n[i];
        M.begin = begin;
        const int bs = Q.blocks[i] < 32 ? 32 : Q.blocks[i];
        M.inv_bs = uint32_t(((1ull << 32) + bs - 1) / bs);
        const long long cells = (long long)(M.base + (M.extra ? 1 : 0)) * bs;
        const int passes = int(((cells + 31) / 32 + kListWarps - 1) / kListWarps);
        if (passes > *warp_passes) *warp_passes = passes;
        if (M.base + (M.extra ? 1 : 0) > *cta_groups) *cta_groups = M.base + (M.extra ? 1 : 0);
        begin += n[i];
    }
    return begin;
}

}  // namespace

cudaError_t launch_gemv_list(const ListDesc& list, int batch, const void* table, cudaStream_t s) {
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    static PerDeviceOnce once;
    e = once.run([] {
        auto set = [](auto kernel) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024); };
        cudaError_t r = set(k_gemv_list<8, true>);
        if (r == cudaSuccess) r = set(k_gemv_list<4, true>);
        if (r == cudaSuccess) r = set(k_gemv_list<8, false>);
        return r;
    });
    if (e != cudaSuccess) return e;
    ListShape Q;
    Q.count = list.count;
    Q.max_blocks = 0;
    ListParams P;
    for (int i = 0; i < list.count; ++i) {
        const Problem& q = list.problems[i];
        ListMatrix& M = P.m[i];
        M.codes = q.codes;
        M.x = static_cast<const __half*>(q.x);
        M.row_scales = q.row_scales;
        M.tail = static_cast<const __half*>(q.tail);
        M.y = q.y;
        M.N = q.N;
        M.K = q.K;
        Q.rows[i] = q.N;
        Q.blocks[i] = (q.tail || q.K % 24 == 0) ? q.K / 24 : (q.K + 23) / 24;
        if (Q.blocks[i] > Q.max_blocks) Q.max_blocks = Q.blocks[i];
    }
    P.batch = batch;
    P.image_cols = Q.max_blocks;
    const DeviceTables* tab = static_cast<const DeviceTables*>(table);
    int passes = 0, groups = 0;
    int grid = split_list(Q, 8, sms, P, &passes, &groups);
    constexpr uint32_t kMaxSmem = 227 * 1024;
    // As few chunks as shared memory allows, of equal size: the rows behind a boundary cost a CTA-wide round of their own
    // (four launches of a 4B layer, whose gate and up matrices come to 136 rows a CTA: 29.7 us with 128 and 8, 27.4 us).
    const uint32_t fixed = list_smem(Q.max_blocks, 0).total, row_bytes = (list_smem(Q.max_blocks, 8).total - fixed) / 8;
    const int room = fixed < kMaxSmem ? int((kMaxSmem - fixed) / row_bytes) & ~7 : 0;
    if (room < kChunkRows) {  // more columns than the shared-memory image can hold
        P.chunk = kChunkRows / 8;
        return launch_pdl(k_gemv_list<8, false>, grid, kListThreads, list_smem(0, kChunkRows).total, s, tab, P);
    }
    auto launch = [&](auto kernel, int R) {
        const int chunks = (groups * R + room - 1) / room;
        P.chunk = (groups + chunks - 1) / chunks;
        return launch_pdl(kernel, grid, kListThreads, list_smem(Q.max_blocks, (P.chunk * R + 7) & ~7).total, s, tab, P);
    };
    // A warp's pass over eight rows is a chain of eight blocks, and every warp runs a whole number of them: half
    // records when their chain is shorter.  A block costs about 82 instructions, a pass about 150 more (record and
    // activations in, row ends): measured on both sides of the line, 12288 x 4096: four passes of eight rows 9.4 us,
    // seven of four 10.2 us; 6144 x 2560: two of eight 6.1 us, three of four 5.6 us.
    const long long chain8 = (long long)passes * (8 * 82 + 150);
    grid = split_list(Q, 4, sms, P, &passes, &groups);
    if ((long long)passes * (4 * 82 + 150) < chain8) return launch(k_gemv_list<4, true>, 4);
    grid = split_list(Q, 8, sms, P, &passes, &groups);
    return launch(k_gemv_list<8, true>, 8);
}

}  // namespace tetra
