// First work of every call with a sparse branch (Eq. 2 on the block mask M), order_lists():
//   - clears the status words the later kernels test (unless the list validator, which then runs
//     before it, has done so),
//   - checks what it reads of the mask anyway: the row offsets of every mask head must be
//     non-negative and non-decreasing; otherwise it records SALAD_ERR_BAD_MASK and the attention
//     kernel of the call returns at once,
//   - writes the launch order of the attention kernel's work items: for every mask head, the query
//     blocks sorted by decreasing length of their kept list, so that the long items start first and
//     the short ones fill the tail.  Counting sort in shared memory; one CTA per mask head.  The
//     order among equal costs is arbitrary (it only affects scheduling).
// Calls with a linear branch run it in CTAs of the state kernel, which needs nothing of it (a launch less, and the
// state pass does not wait for it: 37.1 -> 34.9 us for a call at 12 heads of 2310 tokens, 14.2 -> 11.8 us at the tiny
// configuration, GPU time per call of a replayed graph); work_order_kernel is the form for calls without a state pass.
//
// csr_validate_kernel is the full check of the lists (salad_csr_validate): offsets start at 0, are
// non-decreasing and end within the capacity of col_idx; every row's block ids are strictly
// ascending and inside [0, nKb).  It reads nothing beyond row_ptr[0..rows] and
// col_idx[0..col_capacity), so corrupted lists cannot make it fault.
#pragma once
#include "ptx.cuh"

namespace salad {

constexpr int kOrderBins = 2048;
constexpr int kOrderScratchWords = kOrderBins + 32;      // histogram, then one total per warp

// One CTA of THREADS threads (whole warps) for mask head hm; scratch: kOrderScratchWords words of shared memory, 16-byte aligned.
template <int THREADS>
__device__ __forceinline__ void order_lists(const int32_t* row_ptr, int nQb, int Hm, int hm,
                                            int32_t* order, int32_t* ws_status,
                                            int32_t* user_status, int clear_status, int* scratch) {
    int* hist = scratch;
    int* total = scratch + kOrderBins;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < kOrderBins / 4; i += THREADS) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
    int bad = 0;
    if (hm == 0) {
        // The first CTA is the only writer of the status words here (so a clear can never
        // overtake a report): it checks the offsets of every mask head, eight at a time per thread in flight.
        const long long rows = (long long)Hm * nQb;
        for (long long r0 = tid; r0 < rows; r0 += 8 * THREADS) {
            int a[8], b[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const long long r = r0 + u * THREADS;
                a[u] = r < rows ? row_ptr[r] : 0;
                b[u] = r < rows ? row_ptr[r + 1] : 0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) bad |= (a[u] < 0 || b[u] < a[u]) ? 1 : 0;
        }
    }
    bad = __syncthreads_or(bad);
    if (hm == 0 && tid == 0) {
        if (bad) {
            *ws_status = SALAD_ERR_BAD_MASK;
            if (user_status) *user_status = SALAD_ERR_BAD_MASK;
        } else if (clear_status) {       // (otherwise the list validator, which ran before, owns the words)
            *ws_status = 0;
            if (user_status) *user_status = 0;
        }
    }
    const int32_t* rp = row_ptr + size_t(hm) * nQb;
    // the length of a list, clamped to a bin: a corrupted offset must not index outside the histogram
    // (the order written for a rejected mask is never used: the attention kernel of the call returns at once)
    auto cost_of = [&](int qb) { return max(0, min(kOrderBins - 1, rp[qb + 1] - rp[qb])); };
    for (int qb = tid; qb < nQb; qb += THREADS) atomicAdd(&hist[cost_of(qb)], 1);
    __syncthreads();
    // start position of every cost, largest cost first: an exclusive suffix sum over the bins.  A thread owns PER
    // successive bins, thread 0 the highest; shuffles inside a warp, one total per warp.
    constexpr int PER = (kOrderBins + THREADS - 1) / THREADS;
    const int top = kOrderBins - 1 - tid * PER;                     // this thread's highest bin
    int c[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) { c[i] = top - i >= 0 ? hist[top - i] : 0; sum += c[i]; }
    int incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) total[warp] = incl;
    __syncthreads();
    int start = incl - sum;
    for (int w = 0; w < warp; ++w) start += total[w];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        if (top - i >= 0) hist[top - i] = start;
        start += c[i];
    }
    __syncthreads();
    for (int qb = tid; qb < nQb; qb += THREADS)
        order[size_t(hm) * nQb + atomicAdd(&hist[cost_of(qb)], 1)] = qb;
}

__global__ void __launch_bounds__(1024) work_order_kernel(const int32_t* row_ptr, int nQb, int Hm,
                                                          int32_t* order,
                                                          int32_t* ws_status,
                                                          int32_t* user_status, int clear_status) {
    grid_dependency_wait();           // the kernel before the call, which may have written the lists
    grid_launch_dependents();         // the attention kernel may be placed now; it waits for this one
    __shared__ alignas(16) int scratch[kOrderScratchWords];
    order_lists<1024>(row_ptr, nQb, Hm, blockIdx.x, order, ws_status, user_status, clear_status, scratch);
}

// One warp per CSR row.  The status words (either may be null) receive SALAD_ERR_BAD_MASK when a check
// fails; the host clears them, in stream order, before this kernel.
__global__ void __launch_bounds__(256) csr_validate_kernel(const int32_t* __restrict__ row_ptr,
                                                           const int32_t* __restrict__ col_idx,
                                                           long long col_capacity, int rows, int nKb,
                                                           int32_t* __restrict__ status_a,
                                                           int32_t* __restrict__ status_b) {
    grid_launch_dependents();
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= rows) return;
    const long long a = row_ptr[row], b = row_ptr[row + 1];
    bool bad = (row == 0 && a != 0) || a < 0 || b < a || b > col_capacity;
    if (!bad) {
        for (long long i = a + lane; i < b; i += 32) {
            const int c = col_idx[i];
            if (c < 0 || c >= nKb) bad = true;
            if (i > a && col_idx[i - 1] >= c) bad = true;        // strictly ascending: sorted and unique
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) {
        if (status_a) atomicExch(status_a, SALAD_ERR_BAD_MASK);
        if (status_b) atomicExch(status_b, SALAD_ERR_BAD_MASK);
    }
}

}  // namespace salad
