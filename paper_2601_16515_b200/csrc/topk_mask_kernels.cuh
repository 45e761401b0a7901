// Dynamic Top-K block mask (Appendix A.1, Steps 1-2): per (batch, head) and query block, the k key
// blocks whose mean has the largest average similarity with the block's queries,
//     s[i][j] = < mean of query block i , mean of key block j > ,
// written as the CSR lists the attention kernel consumes (every row keeps kk = min(k, nKb) blocks,
// ascending; a tie goes to the lower block index).
//
//   block_mean_kernel   HBM-bound: Q and K are read once (4*N*d bytes per head).  One CTA per token
//                       block; a thread owns one 16-byte channel group of every G-th row, so a warp
//                       instruction reads 512 contiguous bytes; the row groups are added in a fixed
//                       order through shared memory (deterministic), fp32.
//                       (block_mean_pair_kernel: blocks of 128 queries and 64 keys, the 128 tokens of a
//                       query block and its two key blocks in one CTA with every load in flight at once.)
//   topk_score_kernel   s for a 32 x 128 tile of (query block, key block) pairs per CTA: register-tiled
//                       fp32 FMAs, two at a time, in channel order from channel-major shared memory; the scores
//                       go to the workspace as order-preserving 32-bit images.
//   topk_pick_warp_kernel  per query block (a warp each, the scores in its registers): the kk-th largest score by
//                       bisection on the bits of its image, then an ordered compaction into the CSR row.
//                       (topk_pick_kernel: the same with the scores re-read in every pass, for rows of more
//                       than 2048 key blocks.)
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ptx.cuh"

namespace salad {

constexpr int kMeanThreads = 256;

struct MeanJob {
    const uint4* x;      // bf16 [BH][N][d]
    float* mean;         // fp32 [BH][nB][d], or channel-major [BH][d][ld] when ld > 0
    int block, nB;       // tokens per block, blocks per head
    int ld;              // 0: block-major rows of d channels; > 0: channel-major rows of ld blocks
};

// grid (max nB, BH, 2): z selects the job (queries / keys)
__global__ void __launch_bounds__(kMeanThreads)
block_mean_kernel(MeanJob jq, MeanJob jk, int N, int d)
{
    const MeanJob job = (blockIdx.z == 0) ? jq : jk;
    const int blk = blockIdx.x, bh = blockIdx.y;
    if (blk >= job.nB) return;
    __shared__ float part[kMeanThreads / 8][8 * 16 + 1];      // [row group][channel] (d <= 128)
    const int chunks = d / 8;                                 // 16-byte groups per row: 8 or 16
    const int groups = kMeanThreads / chunks;                 // row groups: 32 or 16
    const int tid = threadIdx.x, c = tid % chunks, g = tid / chunks;
    const int n0 = blk * job.block, n1 = min(N, n0 + job.block);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const uint4* base = job.x + (size_t(bh) * N) * chunks + c;
#pragma unroll 8
    for (int n = n0 + g; n < n1; n += groups) {               // this thread's rows, in token order
        const uint4 v = __ldg(base + size_t(n) * chunks);
        const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(h[e]);
            acc[2 * e] += f.x; acc[2 * e + 1] += f.y;
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) part[g][c * 8 + e] = acc[e];
    __syncthreads();
    if (tid < d) {
        float s = 0.f;
        for (int gg = 0; gg < groups; ++gg) s += part[gg][tid];      // fixed order
        const float m = s / float(n1 - n0);
        if (job.ld > 0) job.mean[(size_t(bh) * d + tid) * job.ld + blk] = m;
        else            job.mean[(size_t(bh) * job.nB + blk) * d + tid] = m;
    }
}

// Blocks of 128 queries and 64 keys: grid (nQb, BH), 256 threads.  The CTA of query block i also takes the key blocks 2i and
// 2i + 1, so all of its 2 * 128 rows are the same token range, and every thread issues all of its loads (8 or 4 rows of Q and
// as many of K) ahead of the adds, half as many CTAs as token blocks with twice the bytes each: 44 -> 39 us at 12 heads of
// 32760 tokens, d = 128 (5.2 TB/s).  The sums run in the same order as in block_mean_kernel.  It lets the score kernel go
// only by its end: score CTAs placed early took shared memory from this kernel's (63 -> 73 us per call).
template <int CHUNKS>                                             // 16-byte groups per row: d / 8
__global__ void __launch_bounds__(kMeanThreads)
block_mean_pair_kernel(const uint4* __restrict__ q, const uint4* __restrict__ k, float* __restrict__ qmean,
                       float* __restrict__ kmeanT, int N, int nQb, int nKb, int ldk)
{
    constexpr int D = CHUNKS * 8, GROUPS = kMeanThreads / CHUNKS, ROWS = 128 / GROUPS, HALF = ROWS / 2;
    __shared__ float part[3][GROUPS][D + 4];                     // queries, keys of block 2i, of block 2i + 1
    const int blk = blockIdx.x, bh = blockIdx.y, tid = threadIdx.x, c = tid % CHUNKS, g = tid / CHUNKS;
    const int n0 = blk * 128;
    const size_t base = (size_t(bh) * N) * CHUNKS + c;
    uint4 vq[ROWS], vk[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int n = n0 + g + r * GROUPS;
        vq[r] = n < N ? __ldg(q + base + size_t(n) * CHUNKS) : make_uint4(0, 0, 0, 0);
        vk[r] = n < N ? __ldg(k + base + size_t(n) * CHUNKS) : make_uint4(0, 0, 0, 0);
    }
    float sum[3][8];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int e = 0; e < 8; ++e) sum[j][e] = 0.f;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const __nv_bfloat162* hq = reinterpret_cast<const __nv_bfloat162*>(&vq[r]);
        const __nv_bfloat162* hk = reinterpret_cast<const __nv_bfloat162*>(&vk[r]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 fq = __bfloat1622float2(hq[e]), fk = __bfloat1622float2(hk[e]);
            sum[0][2 * e] += fq.x; sum[0][2 * e + 1] += fq.y;
            sum[r < HALF ? 1 : 2][2 * e] += fk.x; sum[r < HALF ? 1 : 2][2 * e + 1] += fk.y;
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        *reinterpret_cast<float4*>(&part[j][g][c * 8]) = make_float4(sum[j][0], sum[j][1], sum[j][2], sum[j][3]);
        *reinterpret_cast<float4*>(&part[j][g][c * 8 + 4]) = make_float4(sum[j][4], sum[j][5], sum[j][6], sum[j][7]);
    }
    __syncthreads();
    for (int i = tid; i < 3 * D; i += kMeanThreads) {
        const int j = i / D, ch = i % D;
        const int first = j == 2 ? n0 + 64 : n0, tokens = min(N, first + (j == 0 ? 128 : 64)) - first;
        if (tokens <= 0) continue;                               // the second key block may lie past the end
        float s = 0.f;
#pragma unroll
        for (int gg = 0; gg < GROUPS; ++gg) s += part[j][gg][ch];            // fixed order
        const float m = s / float(tokens);
        if (j == 0) qmean[(size_t(bh) * nQb + blk) * D + ch] = m;
        else        kmeanT[(size_t(bh) * D + ch) * ldk + 2 * blk + j - 1] = m;
    }
}

constexpr int kScoreRows = 32;        // query blocks per CTA (four warps, eight each)
constexpr int kScoreTile = 128;       // key blocks per CTA (four per lane)

// fp32 -> uint32 such that a < b  <=>  image(a) < image(b)  (for non-NaN a, b; -0 is stored as +0)
__device__ __forceinline__ uint32_t ordered_bits(float s) {
    const uint32_t u = __float_as_uint(s + 0.0f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ void cp_async_16(void* smem_dst, const void* gmem_src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst))), "l"(gmem_src) : "memory");
}

constexpr int kScoreChunk = 32;       // channels per shared-memory stage
constexpr int kScoreSmemBytes = 2 * kScoreChunk * (kScoreRows + kScoreTile) * 4;      // two stages: 40 KB

// grid (ceil(nKb / 128), ceil(nQb / 32), BH), 128 threads (an 8 x 4 tile of scores each), 40 KB of dynamic shared memory: two stages of
// 32 channels each, As [32][32] query-block means | Bs [32][128] key-block means, both channel-major; the
// next stage is fetched (asynchronous 16-byte copies) while the current one is multiplied, and five CTAs
// fit on an SM, so the whole grid is resident at once.
//   qmean  [BH][nQb][d]      kmeanT [BH][d][ldk] (ldk a multiple of 128: whole tiles are readable)
//   score  [BH][nQb][nKb]    images of s[i][j] = sum_c qmean[i][c] * kmean[j][c], c ascending
__global__ void __launch_bounds__(128)
topk_score_kernel(const float* qmean, const float* kmeanT, int nQb, int nKb, int ldk,
                  int d, uint32_t* __restrict__ score)
{
    extern __shared__ __align__(16) float sc_smem[];
    constexpr int STAGE = kScoreChunk * (kScoreRows + kScoreTile);       // floats per stage
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j0 = blockIdx.x * kScoreTile, i0 = blockIdx.y * kScoreRows, bh = blockIdx.z;
    grid_dependency_wait();
    grid_launch_dependents();
    const float* ksrc = kmeanT + size_t(bh) * d * ldk + j0;
    const int r_q = tid % kScoreRows, ii = min(i0 + r_q, nQb - 1);
    const float* qsrc = qmean + (size_t(bh) * nQb + ii) * d;
    auto fetch = [&](int chunk, int stage) {
        float* Bs = sc_smem + stage * STAGE + kScoreChunk * kScoreRows;
        const int c0 = chunk * kScoreChunk;
        // key-block means: rows of 128 contiguous floats per channel
        for (int idx = tid; idx < kScoreChunk * (kScoreTile / 4); idx += 128) {
            const int c = idx / (kScoreTile / 4), f = idx % (kScoreTile / 4);
            cp_async_16(Bs + c * kScoreTile + f * 4, ksrc + size_t(c0 + c) * ldk + f * 4);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // query-block means, transposed on the way in: this thread's row, two float4 of channels, in registers while the
    // chunk before them is multiplied (stored at once they left an L2 round trip exposed per chunk)
    constexpr int QV = kScoreChunk / 4 / (128 / kScoreRows);
    float4 qnext[QV];
    auto fetch_q = [&](int chunk) {
#pragma unroll
        for (int e = 0; e < QV; ++e)
            qnext[e] = __ldcg(reinterpret_cast<const float4*>(qsrc + chunk * kScoreChunk) + tid / kScoreRows + e * (128 / kScoreRows));
    };
    auto store_q = [&](int stage) {
        float* As = sc_smem + stage * STAGE;
#pragma unroll
        for (int e = 0; e < QV; ++e) {
            const int c = (tid / kScoreRows + e * (128 / kScoreRows)) * 4;
            As[(c + 0) * kScoreRows + r_q] = qnext[e].x; As[(c + 1) * kScoreRows + r_q] = qnext[e].y;
            As[(c + 2) * kScoreRows + r_q] = qnext[e].z; As[(c + 3) * kScoreRows + r_q] = qnext[e].w;
        }
    };
    // two query rows in one packed accumulator: 16 packed FMAs per channel instead of 32 (the same roundings)
    uint64_t acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[r][u] = pack_f32x2(0.f, 0.f);
    const int chunks = d / kScoreChunk;
    fetch(0, 0);
    fetch_q(0);
    store_q(0);
    for (int ch = 0; ch < chunks; ++ch) {
        if (ch + 1 < chunks) {
            fetch(ch + 1, (ch + 1) & 1);
            fetch_q(ch + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float* As = sc_smem + (ch & 1) * STAGE;
        const float* Bs = As + kScoreChunk * kScoreRows;
#pragma unroll 8
        for (int c = 0; c < kScoreChunk; ++c) {                    // channel order
            const float4 qa = *reinterpret_cast<const float4*>(As + c * kScoreRows + warp * 8);
            const float4 qb = *reinterpret_cast<const float4*>(As + c * kScoreRows + warp * 8 + 4);
            const float4 k4 = *reinterpret_cast<const float4*>(Bs + c * kScoreTile + lane * 4);
            const uint64_t qv[4] = {pack_f32x2(qa.x, qa.y), pack_f32x2(qa.z, qa.w), pack_f32x2(qb.x, qb.y), pack_f32x2(qb.z, qb.w)};
            const uint64_t kv[4] = {pack_f32x2(k4.x, k4.x), pack_f32x2(k4.y, k4.y), pack_f32x2(k4.z, k4.z), pack_f32x2(k4.w, k4.w)};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[r][u] = fma_f32x2(qv[r], kv[u], acc[r][u]);
        }
        if (ch + 1 < chunks) store_q((ch + 1) & 1);
        __syncthreads();                                           // the stage is fetched into again two chunks on
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int i = i0 + warp * 8 + r;
        if (i >= nQb) break;
        uint32_t* out = score + (size_t(bh) * nQb + i) * nKb + j0 + lane * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float lo, hi;
            unpack_f32x2(acc[r / 2][u], lo, hi);
            if (j0 + lane * 4 + u < nKb) out[u] = ordered_bits((r & 1) ? hi : lo);
        }
    }
}

// grid ceil(rows_total / 8), 128 threads: a warp selects for two consecutive rows (query blocks) at
// a time: the kk-th largest score by bisection on the 32 bits of its image (32 counting passes,
// whatever kk), everything above it, and of the scores equal to it the lowest block indices -- the
// same set as kk rounds of "largest remaining, ties to the lower index".
// The lane's share of a row is re-read (from L1/L2) in every pass: this is the kernel for rows too long for
// topk_pick_warp_kernel below (more than 2048 key blocks).
__global__ void __launch_bounds__(128)
topk_pick_kernel(const uint32_t* score, int nKb, int kk, int32_t* __restrict__ row_ptr,
                 int32_t* __restrict__ col_idx, long long rows_total)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    grid_dependency_wait();
    grid_launch_dependents();
    {
        const long long ra = ((long long)blockIdx.x * 4 + warp) * 2;
        if (ra >= rows_total) return;
        const bool two = ra + 1 < rows_total;
        const uint32_t* ka = score + ra * nKb;
        const uint32_t* kb = ka + (two ? nKb : 0);
        // image of the kk-th largest score: the largest T with #{key >= T} >= kk.  (Absent
        // entries are 0 and every candidate is > 0, so they are never counted.)
        uint32_t Ta = 0, Tb = 0;
        for (int bit = 31; bit >= 0; --bit) {
            const uint32_t ca = Ta | (1u << bit), cb = Tb | (1u << bit);
            int na = 0, nb = 0;
            for (int j = lane; j < nKb; j += 32) { na += (ka[j] >= ca) ? 1 : 0; nb += (kb[j] >= cb) ? 1 : 0; }
            na = __reduce_add_sync(0xffffffffu, na); nb = __reduce_add_sync(0xffffffffu, nb);
            if (na >= kk) Ta = ca;
            if (nb >= kk) Tb = cb;
        }
        for (int e = 0; e < (two ? 2 : 1); ++e) {
            const uint32_t* kr = e ? kb : ka;
            const uint32_t T = e ? Tb : Ta;
            int n_gt = 0;
            for (int j = lane; j < nKb; j += 32) n_gt += (kr[j] > T) ? 1 : 0;
            n_gt = __reduce_add_sync(0xffffffffu, n_gt);
            const int need_eq = kk - n_gt;                     // of the scores equal to T, the first need_eq
            // ordered compaction
            const long long row = ra + e;
            int32_t* out = col_idx + row * kk;
            int count = 0, eq_seen = 0;
            for (int j0 = 0; j0 < nKb; j0 += 32) {
                const int j = j0 + lane;
                const uint32_t v = (j < nKb) ? kr[j] : 0u;
                const bool eq = (j < nKb) && v == T;
                const unsigned m_eq = __ballot_sync(0xffffffffu, eq);
                const int my_eq = eq_seen + __popc(m_eq & ((1u << lane) - 1u));
                const bool take = (j < nKb) && (v > T || (eq && my_eq < need_eq));
                const unsigned m = __ballot_sync(0xffffffffu, take);
                if (take) out[count + __popc(m & ((1u << lane) - 1u))] = j;
                count += __popc(m); eq_seen += __popc(m_eq);
            }
            if (lane == 0) {
                row_ptr[row] = int32_t(row * kk);
                if (row == rows_total - 1) row_ptr[rows_total] = int32_t(rows_total * kk);
            }
        }
    }
}

// One warp per row, the row's keys in its registers (key j = lane + 32 i in register i; absent ones 0, every real image is
// > 0).  Nothing crosses warps, so there is no barrier; a pass of the bisection is KPT compares and one warp-wide sum.
//   1. bisection on the bits of the image, from the highest bit in which the row's largest and smallest keys
//      differ: T grows as long as at least kk keys are >= T.  As soon as exactly kk are, the set is known: with
//      distinct scores after about half of the passes.
//      (A CTA per row with radix passes over shared-memory histograms, which this replaces, took 13 us for 3072 rows of
//      512 scores against 11, and nothing fitted it beyond 1024: 8 heads of 75600 tokens, 259 -> 161 us per call.)
//   2. ordered compaction with a ballot per 32 keys; of the keys equal to T only as many as are missing, the lowest
//      indices first (a tie goes to the lower block index).
template <int KPT>
__global__ void __launch_bounds__(128)
topk_pick_warp_kernel(const uint32_t* score, int nKb, int kk, int32_t* __restrict__ row_ptr,
                      int32_t* __restrict__ col_idx, long long rows_total)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * 4 + warp;
    grid_dependency_wait();
    grid_launch_dependents();
    if (row >= rows_total) return;
    const uint32_t* kr = score + row * nKb;
    uint32_t key[KPT], lo = 0xffffffffu, hi = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const bool in = lane + 32 * i < nKb;
        key[i] = in ? __ldcg(kr + lane + 32 * i) : 0u;
        if (in) { lo = min(lo, key[i]); hi = max(hi, key[i]); }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const int top = 31 - __clz(lo ^ hi);                    // -1: all keys are the same
    uint32_t T = top < 0 ? lo : (lo & ~((2u << top) - 1u)); // what all of them have in common: nKb >= kk keys are >= T
    int at_least = nKb;
    for (int bit = top; bit >= 0 && at_least != kk; --bit) {
        const uint32_t c = T | (1u << bit);
        int n = 0;
#pragma unroll
        for (int i = 0; i < KPT; ++i) n += (key[i] >= c) ? 1 : 0;
        n = __reduce_add_sync(0xffffffffu, n);
        if (n >= kk) { T = c; at_least = n; }
    }
    // at_least keys are >= T.  More than kk: T is the kk-th largest image itself and the surplus is among the equal ones.
    int need_eq = nKb;
    if (at_least > kk) {
        int n = 0;
#pragma unroll
        for (int i = 0; i < KPT; ++i) n += (key[i] > T) ? 1 : 0;
        need_eq = kk - __reduce_add_sync(0xffffffffu, n);
    }
    int32_t* out = col_idx + row * kk;
    const unsigned below = (1u << lane) - 1u;
    int count = 0, eq_seen = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const bool in = lane + 32 * i < nKb;
        bool take = in && key[i] >= T;
        if (at_least > kk) {
            const bool eq = in && key[i] == T;
            const unsigned m_eq = __ballot_sync(0xffffffffu, eq);
            if (eq && eq_seen + __popc(m_eq & below) >= need_eq) take = false;
            eq_seen += __popc(m_eq);
        }
        const unsigned m = __ballot_sync(0xffffffffu, take);
        if (take) out[count + __popc(m & below)] = lane + 32 * i;
        count += __popc(m);
    }
    if (lane == 0) {
        row_ptr[row] = int32_t(row * kk);
        if (row == rows_total - 1) row_ptr[rows_total] = int32_t(rows_total * kk);
    }
}

}  // namespace salad
