// Block-sparse softmax attention (Eq. 2) fused with the apply step of ReLU linear attention
// (Eq. 3) and the scaled residual sum of Algorithm 1, for sm_100a.
//
// One CTA owns one query block of one (batch, head): a 128-row MMA tile.  Two CTAs share an SM
// (each takes half of its shared memory, registers and tensor memory), so the set-up, the first
// loads and the epilogue of one overlap the main loop of the other, and the two tiles of an SM run
// independently of each other.
//   warp 0        TMA producer of the Q tile, the K ring and (at the end) the linear-state tile
//   warp 1        TMA producer of the V ring (independent of the K ring, so neither ring can
//                 stall the other); stores the output tile, which is staged over that ring
//   warp 2        tcgen05 issuer of S = Q K^T; owns the TMEM allocation
//   warp 3        tcgen05 issuer of O += P V and of the linear numerator
//                 (an issuing warp walks its loop as a whole, every lane polling the barriers, and one
//                 elected lane issues: the operands of a product are then warp-uniform values, which
//                 keeps the cost of issuing one low -- measured 27 against 45 cycles per instruction
//                 when a single lane runs the loop alone)
//   warps 4-11    softmax + epilogue warps: a warp works on 16 query rows (TMEM lanes) with the
//                 16-lane load/store shapes, four threads share a row and each thread serves two
//                 rows; row maxima and sums are combined with two shuffles
// Masked blocks are never loaded.
//
// S = Q K^T (128x64xd, operands in shared memory) of block t lands in TMEM score buffer t & 1;
// the softmax warps copy it to registers and write P = exp2(.), as bf16, over the first half of
// the same buffer, which O += P V then reads.  The scores of block t + 1 go to the other buffer
// as soon as the P V product of block t - 1 has read it, so both products of the neighbouring
// blocks overlap the softmax of block t.  The running max lives in the log2 domain; exponentials
// are formed against the max of the earlier blocks without looking at the block's own, and only when
// a thread's 16 probabilities of a row sum to more than 2^12 are the scores read again, their maxima formed and the O
// accumulator brought to the new max.  (P, l and O are floating-point numbers with a factor in common: 2^12 in it
// changes none of their relative errors.)  The block maxima and the vote on them were a sixth of the softmax
// arithmetic; without them the launch is 2 % shorter and takes 2 % less energy, which is what counts at the power
// limit (12 heads of 32760 tokens, back to back: 659 -> 646 us at 90 % sparsity, 5870 -> 5760 us with all blocks
// kept, d = 64: 490 -> 477 us).  The two products have their own issuing warps: each waits only for
// what its next MMA series needs, so it reacts as soon as that arrives.  One commit per series: the
// barrier that announces the scores of block t also frees the K-ring stage for block t + 2, the one
// that announces the completion of P V the V-ring stage.
// Every warp has the 80 registers of the launch (d = 64 takes 75; at d = 128 one word of the epilogue is on the stack).  The producer
// and issuer warps need fewer, but none are handed to the softmax warps (setmaxnreg): compiled with that instruction, forms of this
// kernel lost values that live across it, without a word from the compiler -- with 32 against 104 registers the head's index in the
// storing warp (every tile went to the first head), with 48 against 96 the list's length in the softmax warps (the
// softmax part was left out) -- and the same sources without it are right.  Nor does a CTA take over further items of the grid (cluster
// launch control): with the loop over items around it the softmax loop wants 96 registers, 80 cost it 3 % (11.06 -> 11.48 ms with
// all blocks kept at 2 x 12 heads of 32760 tokens); with them, calls of short lists gained by it (12 + 12 heads of 32760 tokens
// at 95 % 795 -> 780 us) about what calls of few items and long lists lost (2 heads of 35496 tokens, d = 64, all blocks kept, 847 -> 999).
// After the last block the softmax warps apply ReLU to the Q rows in shared memory and compute the
// linear denominator with plain FMAs; the linear state (bf16, transposed) is loaded over the K
// ring, which is idle by then; the issuing thread multiplies ReLU(Q) with it, and the epilogue
// writes
//     O = O_acc / l + (s_b lambda_h / (den + eps)) * num
// once, as bf16, through a TMA store.
// The kernels that make the linear state come before this one in the stream and run beside it: this
// kernel is launched to start early and waits for them only in warp 0, just before the state tile and
// the normaliser Z are fetched, so the softmax attention of the first tiles hides the state pass.
//
// TMEM columns (256 allocated):  [0,64) and [64,128) two score buffers (block t uses buffer
// t & 1; its probabilities, packed bf16, overwrite the first 32 columns of the same buffer);
// [128,128+D) O.  The linear numerator reuses [0,D).
#pragma once
#include <type_traits>

#include "ptx.cuh"

namespace salad {

enum FusedMode { MODE_SPARSE = 1, MODE_LINEAR = 2, MODE_FUSED = 3 };

// Heads with temporal locality (Appendix A.1): their tokens are taken in the order that groups them by spatial
// position, m = s * T + t for token n = t * S + s, through 4-D tensor maps, without a re-ordering pass.  A
// key block of such a head is the T tokens of ks spatial positions (ks * T <= 64 rows of the 64-row tile), a
// query block those of kq positions (kq * T <= 128 rows); the unused rows of the tiles hold zeros and their
// keys are masked.
struct TemporalHeads {
    int T, S;                    // T == 0: no head is re-ordered
    int kq, ks;                  // spatial positions per query / key block
    int nQb, nKb;                // blocks per head: ceil(S / kq), ceil(S / ks)
    uint32_t flags[8];           // bit h: head h is temporal (H <= 256)
};

struct FusedParams {
    int N, H, nQb, nKb, Bq, Hm, mode;     // nQb: list rows per mask head; nKb: key blocks of a head in token order
    int nQb_tok;                 // query blocks of a head in token order (== nQb unless temporal heads have more)
    TemporalHeads th;
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const int32_t* order;        // [Hm][nQb] launch order of the query blocks, or null (identity)
    int BH;                      // batch * heads
    int by_rank;                 // order of the work items: 1: by expense over all heads, 0: head by head
    const float* static_scale;   // [H] or null (=1)
    const float* dyn_scale;      // [B] or null (=1)
    const float* z;              // [B*H, D] linear normaliser state
    float* lse;                  // optional [B*H, N]
    float scale_log2;            // softmax_scale * log2(e)
    float eps;
    float drop_tau;              // linear branch of batch item b skipped when dyn_scale[b] < drop_tau
    const __half* rope;          // [N][D] fp16: (cos, sin) per token and channel pair of the rotary linear branch, or null
    int wait_at_top;             // 1: wait for the kernel before this one at once (calls without state kernels)
    int32_t* ws_status;          // library status word (never null)
    int32_t* user_status;        // optional
};

template <int D>
struct FusedCfg {
    static constexpr int BK = 64;
    static constexpr int CH = D / 64;               // 128-byte chunks per row
    static constexpr int Q_CHUNK = 128 * 128;       // bytes of one 64-column chunk of the Q tile
    static constexpr int Q_BYTES = CH * Q_CHUNK;
    static constexpr int KV_CHUNK = BK * 128;
    static constexpr int KV_BYTES = CH * KV_CHUNK;  // one K or V tile
    static constexpr int ST_CHUNK = D * 128;
    static constexpr int ST_BYTES = CH * ST_CHUNK;  // linear state, bf16 [D][D]: as large as the K ring
    static constexpr int NK = 2, NV = 2;
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = Q_BYTES;
    static constexpr int OFF_ST = OFF_K;            // loaded over the K ring once every Q K^T has completed
    static constexpr int OFF_V = OFF_K + NK * KV_BYTES;
    static constexpr int SMEM_BYTES = OFF_V + NV * KV_BYTES + 1024;   // + alignment slack: 97 KB at D = 128
    static constexpr int THREADS = 384;
    // TMEM columns: two score buffers of 64 (P overwrites the first 32 columns of the buffer its
    // scores came from), then the output accumulator
    static constexpr uint32_t COL_SP = 0, SP_STRIDE = 64, COL_O = 128;
    static constexpr uint32_t TMEM_COLS = 256;
};
static_assert(FusedCfg<128>::ST_BYTES == FusedCfg<128>::NK * FusedCfg<128>::KV_BYTES, "the state tile fills the K ring");
static_assert(FusedCfg<64>::ST_BYTES <= FusedCfg<64>::NK * FusedCfg<64>::KV_BYTES, "the state tile fits in the K ring");

struct FusedBarriers {
    uint64_t q_full, st_full, k_full[2], v_full[2];
    uint64_t s_full[2], p_ready[2], pv_done[2], o_final, lin_ready, lin_done, out_staged, z_full;
};

// A work item: a query block of a (batch, head) with its kept list.
struct FusedItem {
    int qb, bh, ls, len;
    int linear;                        // it has a linear branch,
    float scale;                       // scaled by this
};

template <int D>
__global__ void __launch_bounds__(384, 2)
salad_fused_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o,
                   const __grid_constant__ CUtensorMap map_st, const __grid_constant__ CUtensorMap map_q4,
                   const __grid_constant__ CUtensorMap map_k4, const __grid_constant__ CUtensorMap map_v4,
                   const __grid_constant__ CUtensorMap map_o4, const FusedParams p)
{
    using C = FusedCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ FusedBarriers bars;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    __shared__ alignas(16) float z_s[D];          // linear normaliser state of this head

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t s_base = smem_u32(smem);
    const int tid = threadIdx.x, lane = tid & 31;
    // The same as tid >> 5, but known to be the same in every lane, which keeps the roles' branches free of
    // reconvergence code (638 -> 629 us at 12 heads of 32760 tokens, 90 % sparsity, attention alone, at the power limit,
    // 470 -> 451 at d = 64, 35.6 -> 34.7 for 2310 tokens; measured with a register split that is gone).
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    // The work order (and the verdict on the lists) comes from the first kernel of the call.  Without a linear
    // branch that is the kernel before this one.  With one, it is the state kernel, whose ordering CTAs let the kernels
    // after it go only when their results are in the L2; this kernel reads them from there and does not wait for
    // the state kernels here: it runs beside them and waits only where it first touches the state, in the epilogue.
    if ((p.mode & MODE_LINEAR) == 0 || p.wait_at_top) grid_dependency_wait();
    grid_launch_dependents();

    // Work items: head by head, within a head the query blocks from the most to the least expensive, so that the
    // kernel ends on short items and K/V of one head stay hot in L2; or, where K and V of all heads fit there (by_rank),
    // the most expensive item of every head, then the next of every head: the CTAs that wait for a state CTA's place, and the second
    // CTA of an SM where the items do not fill all, then hold cheap items, and the launch ends on the cheapest of all heads.
    const FusedItem item = [&](int block) {
        FusedItem it;
        const int rank = p.by_rank ? block / p.BH : block % p.nQb;
        it.bh = p.by_rank ? block % p.BH : block / p.nQb;
        const int h = it.bh % p.H, b = it.bh / p.H;
        const int hm = (p.Hm == 1) ? 0 : (p.Hm == p.H ? h : it.bh);   // one mask, one per head, or one per (batch, head)
        it.qb = p.order ? __ldcg(p.order + size_t(hm) * p.nQb + rank) : rank;
        it.linear = (p.mode & MODE_LINEAR) != 0;
        it.scale = 1.f;
        if (it.linear) {
            if (p.static_scale) it.scale *= __ldg(p.static_scale + h);
            if (p.dyn_scale) {
                const float dyn = __ldg(p.dyn_scale + b);
                it.scale *= dyn;
                if (dyn < p.drop_tau) it.linear = 0;       // post-tuning branch dropping (Sec. 4.3): no linear work at all for a dropped batch item
            }
        }
        it.ls = 0; it.len = 0;
        if ((p.mode & MODE_SPARSE) != 0) {                               // kept list of the query block
            it.ls = __ldg(p.row_ptr + size_t(hm) * p.nQb + it.qb);
            it.len = __ldg(p.row_ptr + size_t(hm) * p.nQb + it.qb + 1) - it.ls;
        }
        return it;
    }(blockIdx.x);
    const int qb = item.qb, bh = item.bh, len = item.len;
    const bool linear = item.linear != 0;
    // temporal head: blocks of spatial positions, fetched through the 4-D maps
    const int h0 = bh % p.H;
    const bool perm = p.th.T > 0 && ((p.th.flags[h0 >> 5] >> (h0 & 31)) & 1u);
    const int q_rows = perm ? p.th.kq * p.th.T : p.Bq;          // rows of the 128-row tile that hold queries
    const int k_rows = perm ? p.th.ks * p.th.T : C::BK;         // rows of a 64-row tile that hold keys
    if (qb >= (perm ? p.th.nQb : p.nQb_tok)) return;       // (a list row beyond this head's blocks: whole CTA)

    // softmax warps whose 16 rows hold queries (64-row query blocks: four of the eight); the others do nothing
    const int row_warps = (q_rows + 15) >> 4;

    // ------------------------------------------------------------------ set-up
    if (tid == 0) {
        // 2: an earlier kernel of this call has already reported a failure (a rejected mask, an expired wait):
        // this CTA starts nothing and reports nothing; 1 (set by a bounded wait of this CTA): a time-out
        abort_flag = (*reinterpret_cast<volatile int32_t*>(p.ws_status) != 0) ? 2 : 0;
        mbar_init(smem_u32(&bars.q_full), 1);
        mbar_init(smem_u32(&bars.st_full), 1);
        mbar_init(smem_u32(&bars.o_final), 1);
        mbar_init(smem_u32(&bars.lin_ready), row_warps);
        mbar_init(smem_u32(&bars.lin_done), 1);
        mbar_init(smem_u32(&bars.out_staged), row_warps);
        mbar_init(smem_u32(&bars.z_full), 32);
        for (int j = 0; j < 2; ++j) {
            mbar_init(smem_u32(&bars.s_full[j]), 1);
            mbar_init(smem_u32(&bars.p_ready[j]), row_warps);  // one arrival per softmax warp
            mbar_init(smem_u32(&bars.pv_done[j]), 1);
            mbar_init(smem_u32(&bars.k_full[j]), 1);
            mbar_init(smem_u32(&bars.v_full[j]), 1);
        }
        fence_mbar_init();
    }
    if (q_rows < 128 || k_rows < C::BK) {
        // rows [q_rows, 128) of the Q tile and [k_rows, 64) of the K and V tiles are never written by TMA:
        // zero them so that the unused part of an MMA tile holds finite numbers (zero keys are masked, zero
        // value rows meet zero probabilities)
        for (int i = tid; i < C::CH * (128 - q_rows) * 8; i += C::THREADS) {
            const int chunk = i / ((128 - q_rows) * 8), rest = i % ((128 - q_rows) * 8);
            *reinterpret_cast<uint4*>(smem + C::OFF_Q + chunk * C::Q_CHUNK + q_rows * 128 + rest * 16) =
                make_uint4(0, 0, 0, 0);
        }
        const int per_tile = (C::BK - k_rows) * 8;                // 16-byte vectors per 64-row chunk of a K or V tile
        for (int i = tid; i < (C::NK + C::NV) * C::CH * per_tile; i += C::THREADS) {
            const int tile = i / per_tile, rest = i % per_tile;  // K: [chunk][stage], V: [stage][chunk]: all 8 KB apart
            *reinterpret_cast<uint4*>(smem + C::OFF_K + tile * C::KV_CHUNK + k_rows * 128 + rest * 16) = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async_smem();
    }
    if (warp == 2) { tmem_alloc(smem_u32(&tmem_base_slot), C::TMEM_COLS); tmem_relinquish(); }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_base_slot;
    volatile int* abortp = &abort_flag;
    const bool inherited_abort = abort_flag != 0;      // uniform: read after the barrier above, before any wait

    // a bounded wait taken by a whole warp: warp-uniform outcome
    auto wait_warp = [&](uint64_t* bar, uint32_t parity) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity, abortp));
    };
    if (!inherited_abort) {
    if (warp < 4) {
    if (warp == 0) {
        // ============================================================== TMA producer: Q, the K ring, the state tile
        bool ok = true;
        if (lane == 0) {
            // A block with no kept key block and no linear branch never reads Q.
            if (len > 0 || linear) {
                const uint32_t bar = smem_u32(&bars.q_full);
                mbar_arrive_expect_tx(bar, uint32_t(q_rows) * D * 2);
                for (int ch = 0; ch < C::CH; ++ch) {
                    if (perm) tma_load_4d(s_base + C::OFF_Q + ch * C::Q_CHUNK, &map_q4, bar, ch * 64, 0, qb * p.th.kq, bh);
                    else tma_load_3d(s_base + C::OFF_Q + ch * C::Q_CHUNK, &map_q, bar, ch * 64, qb * p.Bq, bh);
                }
            }
            prefetch_tmap(&map_k);
            int col = len > 0 ? __ldg(p.col_idx + item.ls) : 0;
            for (int t = 0; t < len; ++t) {
                const int s = t & 1;
                // stage s is free once Q K^T of the block before the last has completed: the barrier that hands its
                // scores to the softmax warps says so (one commit serves both)
                if (t >= C::NK) ok = mbar_wait(smem_u32(&bars.s_full[s]), ((t >> 1) - 1) & 1, abortp);
                if (!ok) break;
                const uint32_t bar = smem_u32(&bars.k_full[s]);
                mbar_arrive_expect_tx(bar, uint32_t(k_rows) * D * 2);
                for (int ch = 0; ch < C::CH; ++ch) {     // chunk-major: the two stages of a chunk are adjacent
                    const uint32_t dst = s_base + C::OFF_K + ch * (C::NK * C::KV_CHUNK) + s * C::KV_CHUNK;
                    if (perm) tma_load_4d(dst, &map_k4, bar, ch * 64, 0, col * p.th.ks, bh);
                    else tma_load_3d(dst, &map_k, bar, ch * 64, col * C::BK, bh);
                }
                if (t + 1 < len) col = __ldg(p.col_idx + item.ls + t + 1);
            }
        }
        if (linear) {
            // From here on the linear state is needed: wait for the kernels that make it (whole warp: the
            // other lanes fetch the normaliser Z of this head for the softmax warps meanwhile).
            __syncwarp();
            grid_dependency_wait();
            if (*reinterpret_cast<volatile int32_t*>(p.ws_status) != 0 && *abortp == 0) *abortp = 2;   // the state kernel gave up (and said so)
            for (int a = lane; a < D; a += 32) z_s[a] = __ldcg(p.z + size_t(bh) * D + a);
            mbar_arrive(smem_u32(&bars.z_full));
            if (lane == 0 && ok) {
                // the state tile goes over the K ring: every Q K^T must have read its K block.  The products
                // complete in order, so the last one (signalled on its score buffer's barrier) covers all.
                if (len > 0) ok = mbar_wait(smem_u32(&bars.s_full[(len - 1) & 1]), ((len - 1) >> 1) & 1, abortp);
                if (ok) {
                    prefetch_tmap(&map_st);
                    const uint32_t bar = smem_u32(&bars.st_full);
                    mbar_arrive_expect_tx(bar, C::ST_BYTES);
                    for (int ch = 0; ch < C::CH; ++ch)
                        tma_load_3d(s_base + C::OFF_ST + ch * C::ST_CHUNK, &map_st, bar, ch * 64, 0, bh);
                }
            }
        }
    } else if (warp == 1) {
        // ============================================================== TMA producer of the V ring, output store
        if (lane == 0) {
            prefetch_tmap(&map_v);
            bool ok = true;
            for (int t = 0; t < len; ++t) {
                const int s = t & 1;
                // stage s is free once P V of the block before the last has completed
                if (t >= C::NV) ok = mbar_wait(smem_u32(&bars.pv_done[s]), ((t >> 1) - 1) & 1, abortp);
                if (!ok) break;
                const int col = __ldg(p.col_idx + item.ls + t);
                const uint32_t bar = smem_u32(&bars.v_full[s]);
                mbar_arrive_expect_tx(bar, uint32_t(k_rows) * D * 2);
                for (int ch = 0; ch < C::CH; ++ch) {
                    const uint32_t dst = s_base + C::OFF_V + s * C::KV_BYTES + ch * C::KV_CHUNK;
                    if (perm) tma_load_4d(dst, &map_v4, bar, ch * 64, 0, col * p.th.ks, bh);
                    else tma_load_3d(dst, &map_v, bar, ch * 64, col * C::BK, bh);
                }
            }
            // the output tile, staged over the V ring
            if (ok && mbar_wait(smem_u32(&bars.out_staged), 0, abortp)) {
                for (int ch = 0; ch < C::CH; ++ch) {
                    if (perm) tma_store_4d(&map_o4, s_base + C::OFF_V + ch * C::Q_CHUNK, ch * 64, 0, qb * p.th.kq, bh);
                    else tma_store_3d(&map_o, s_base + C::OFF_V + ch * C::Q_CHUNK, ch * 64, qb * p.Bq, bh);
                }
                tma_store_commit();
                // only the shared-memory source must have been read before the CTA exits; the
                // writes are complete, like all of the kernel's, when the grid is
                tma_store_wait_read_all();
            }
        }
    } else if (warp == 2) {
        // ============================================================== issuer of S = Q K^T
        // The whole warp walks the loop (every lane polls the barriers) and one elected lane issues: the
        // operands of the products are then warp-uniform values, which is what keeps the cost of issuing
        // a product low (measured: 27 against 45 cycles per instruction when one lane runs the loop alone).
        const uint32_t idesc_qk = make_idesc_bf16(128, C::BK, 0, 0);
        constexpr uint32_t HI = sdesc_hi_sw128(1024);   // the high descriptor word is one constant here
        const uint32_t q_lo = sdesc_lo(s_base + C::OFF_Q, 16);
        const uint32_t k_lo0 = sdesc_lo(s_base + C::OFF_K, 16);
        bool ok = true;
        if (len > 0) ok = wait_warp(&bars.q_full, 0);
        for (int t = 0; t < len && ok; ++t) {
            const int s = t & 1;
            ok = wait_warp(&bars.k_full[s], (t >> 1) & 1);
            // score buffer s held P of the block before the last: its P V product must have read it
            if (ok && t >= 2) ok = wait_warp(&bars.pv_done[s], ((t >> 1) - 1) & 1);
            if (!ok) break;
            tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t kb_lo = k_lo0 + s * (C::KV_CHUNK >> 4);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)   // 16 channels: 32 bytes of each Q and K row, chunk kk/4
                    mma_ss_lohi(tmem + C::COL_SP + s * C::SP_STRIDE,
                                q_lo + (((kk / 4) * C::Q_CHUNK + (kk % 4) * 32) >> 4), HI,
                                kb_lo + (((kk / 4) * (C::NK * C::KV_CHUNK) + (kk % 4) * 32) >> 4), HI, idesc_qk, kk > 0);
                tc_commit(smem_u32(&bars.s_full[s]));
            }
            __syncwarp();
        }
    } else if (warp == 3) {
        // ============================================================== issuer of O += P V and of the linear numerator
        const uint32_t idesc_pv = make_idesc_bf16(128, D, 0, 1);
        const uint32_t idesc_lin = make_idesc_bf16(128, D, 0, 0);
        constexpr uint32_t HI = sdesc_hi_sw128(1024);
        const uint32_t q_lo = sdesc_lo(s_base + C::OFF_Q, 16);
        const uint32_t v_lo0 = sdesc_lo(s_base + C::OFF_V, C::KV_CHUNK);
        bool ok = true;
        for (int t = 0; t < len && ok; ++t) {
            const int s = t & 1;
            ok = wait_warp(&bars.v_full[s], (t >> 1) & 1);
            if (ok) ok = wait_warp(&bars.p_ready[s], (t >> 1) & 1);
            if (!ok) break;
            tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t vb_lo = v_lo0 + s * (C::KV_BYTES >> 4);
                const uint32_t p_col = tmem + C::COL_SP + s * C::SP_STRIDE;
#pragma unroll
                for (int kk = 0; kk < C::BK / 16; ++kk)      // 16 keys = 16 rows of 128 bytes
                    mma_ts_lohi(tmem + C::COL_O, p_col + kk * 8, vb_lo + ((kk * 2048) >> 4), HI, idesc_pv,
                                (t > 0 || kk > 0) ? 1u : 0u);
                tc_commit(smem_u32(&bars.pv_done[s]));
                if (t + 1 == len) tc_commit(smem_u32(&bars.o_final));
            }
            __syncwarp();
        }
        if (ok && linear) {
            ok = wait_warp(&bars.st_full, 0);
            if (ok) ok = wait_warp(&bars.lin_ready, 0);
            if (ok) {
                tc_fence_after_sync();
                if (elect_one()) {
                    const uint32_t st_lo = sdesc_lo(s_base + C::OFF_ST, 16);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        mma_ss_lohi(tmem, q_lo + (((kk / 4) * C::Q_CHUNK + (kk % 4) * 32) >> 4), HI,
                                    st_lo + (((kk / 4) * C::ST_CHUNK + (kk % 4) * 32) >> 4), HI, idesc_lin, kk > 0);
                    tc_commit(smem_u32(&bars.lin_done));
                }
                __syncwarp();
            }
        }
    }
    } else {
        // ============================================================== softmax + epilogue
        // Eight warps.  A warp works on 16 TMEM lanes (query rows) with the 16-lane
        // load/store shapes: four threads share a row, each holding a quarter of its columns,
        // and every thread serves two rows (a and a + 8).  Row maxima and sums are combined
        // with two shuffles inside the group of four.
        const int sw = warp - 4;
        const int q4 = lane & 3;                                // position in the group of four
        const int lane0 = (warp & 3) * 32 + (sw >> 2) * 16;          // first TMEM lane of this warp
        // (the thread's two query rows: lane0 + lane / 4 and eight more)
        // Without queries in its rows a warp leaves its P as it is: whatever it holds meets only accumulator rows that nobody
        // reads.  (64-row query blocks spend half of the exponentials for nothing otherwise: 12 heads of 32760 tokens
        // 1070 -> 932 us per fused call, 2310 tokens 40.1 -> 38.5.)
        if (lane0 < q_rows) {
        const uint32_t t_tile = tmem + (uint32_t(lane0) << 16);
        // every lane of a warp must take the same path around the warp-collective tcgen05
        // loads/stores, so the outcome of a bounded wait is made warp-uniform
        auto wait_uniform = [&](uint64_t* bar, uint32_t parity) -> bool {
            return __all_sync(0xffffffffu, mbar_wait(smem_u32(bar), parity, abortp));
        };
        auto quad_max = [](float v) -> float {
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
            return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
        };
        auto quad_sum = [](float v) -> float {
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            return v + __shfl_xor_sync(0xffffffffu, v, 2);
        };

        bool ok = true;
        float m_a = -INFINITY, m_b = -INFINITY;                 // running maxima (log2 domain)
        float l_a = 0.f, l_b = 0.f;                             // this thread's share of the row sums
        // Only the last key block of the sequence can be short (N not a multiple of 64), and in an ascending
        // list it can only be the last entry: one look at that entry, before the loop, settles which block
        // needs its missing keys masked.
        // (A temporal head: every block holds ks * T keys, the last one those of the positions that exist.)
        int valid_last = k_rows;
        if (len > 0) {
            if (perm) {
                if (__ldg(p.col_idx + item.ls + len - 1) == p.th.nKb - 1) valid_last = (p.th.S - (p.th.nKb - 1) * p.th.ks) * p.th.T;
            } else if ((p.N % C::BK) != 0 && __ldg(p.col_idx + item.ls + len - 1) == p.nKb - 1) {
                valid_last = p.N - (p.nKb - 1) * C::BK;
            }
        }
        const int limits = valid_last | (k_rows << 8);          // (one register instead of two)
        constexpr float SUM_LIMIT = 4096.f;
        for (int t = 0; t < len && ok; ++t) {
            const int s = t & 1;
            ok = wait_uniform(&bars.s_full[s], (t >> 1) & 1);
            if (!ok) break;
            tc_fence_after_sync();
            uint32_t pk[16];
            bool renew = t == 0;                // form the maxima of this block first
            while (true) {                      // once, or twice when the first pass finds that the max has to move
                // x[4n], x[4n+1] = S(row a, keys 8n + 2 q4, + 1);  x[4n+2], x[4n+3] = the same keys of row b
                uint32_t xr[32];
                tmem_ld_16x256b_x8(t_tile + C::COL_SP + s * C::SP_STRIDE, xr);
                float* x = reinterpret_cast<float*>(xr);
                const int valid = (t + 1 == len) ? (limits & 255) : (limits >> 8);      // keys of this block that exist
                if (valid < C::BK) {
#pragma unroll
                    for (int n = 0; n < 8; ++n) {
                        const int key = 8 * n + 2 * q4;
                        if (key >= valid) { x[4 * n] = -INFINITY; x[4 * n + 2] = -INFINITY; }
                        if (key + 1 >= valid) { x[4 * n + 1] = -INFINITY; x[4 * n + 3] = -INFINITY; }
                    }
                }
                if (renew) {
                    float mxa = fmaxf(x[0], x[1]), mxb = fmaxf(x[2], x[3]);
#pragma unroll
                    for (int n = 1; n < 8; ++n) {
                        mxa = fmaxf(mxa, fmaxf(x[4 * n], x[4 * n + 1]));
                        mxb = fmaxf(mxb, fmaxf(x[4 * n + 2], x[4 * n + 3]));
                    }
                    const float msa = quad_max(mxa) * p.scale_log2, msb = quad_max(mxb) * p.scale_log2;
                    if (t == 0) {
                        m_a = msa; m_b = msb;
                    } else {
                        // The accumulator of this warp's rows is brought to the new max, once the previous P V product
                        // has landed in it.  pv_done[b] completes a phase for every second block; the product of block
                        // t cannot be issued before this warp hands over P of block t, so the barrier is at most one
                        // phase past the one tested here and the parity test is exact.
                        ok = wait_uniform(&bars.pv_done[s ^ 1], ((t - 1) >> 1) & 1);
                        if (!ok) break;
                        tc_fence_after_sync();
                        const float na = fmaxf(m_a, msa), nb = fmaxf(m_b, msb);
                        const float al_a = ex2_approx(m_a - na), al_b = ex2_approx(m_b - nb);
                        l_a *= al_a; l_b *= al_b;
                        m_a = na; m_b = nb;
#pragma unroll 1
                        for (int cc = 0; cc < D / 32; ++cc) {
                            uint32_t orr[16];
                            tmem_ld_16x256b_x4(t_tile + C::COL_O + cc * 32, orr);
#pragma unroll
                            for (int n = 0; n < 4; ++n) {
                                orr[4 * n] = __float_as_uint(__uint_as_float(orr[4 * n]) * al_a);
                                orr[4 * n + 1] = __float_as_uint(__uint_as_float(orr[4 * n + 1]) * al_a);
                                orr[4 * n + 2] = __float_as_uint(__uint_as_float(orr[4 * n + 2]) * al_b);
                                orr[4 * n + 3] = __float_as_uint(__uint_as_float(orr[4 * n + 3]) * al_b);
                            }
                            tmem_st_16x256b_x4(t_tile + C::COL_O + cc * 32, orr);
                        }
                        tmem_wait_st();
                    }
                }
                // P = exp2(x * scale - m), packed bf16: word 2n = row a, keys (8n + 2 q4, + 1) = packed
                // column 4n + q4 of the P tile, word 2n + 1 the same of row b -- the 16x128b layout
                const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2);
                const uint64_t nma = pack_f32x2(-m_a, -m_a), nmb = pack_f32x2(-m_b, -m_b);
                uint64_t acc_a = pack_f32x2(0.f, 0.f), acc_b = acc_a;
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    float a0, a1, b0, b1;
                    unpack_f32x2(fma_f32x2(pack_f32x2(x[4 * n], x[4 * n + 1]), sc2, nma), a0, a1);
                    unpack_f32x2(fma_f32x2(pack_f32x2(x[4 * n + 2], x[4 * n + 3]), sc2, nmb), b0, b1);
                    const float pa0 = ex2_approx(a0), pa1 = ex2_approx(a1), pb0 = ex2_approx(b0), pb1 = ex2_approx(b1);
                    acc_a = add_f32x2(acc_a, pack_f32x2(pa0, pa1));
                    acc_b = add_f32x2(acc_b, pack_f32x2(pb0, pb1));
                    pk[2 * n] = pack_bf16x2(pa0, pa1);
                    pk[2 * n + 1] = pack_bf16x2(pb0, pb1);
                }
                float sa0, sa1, sb0, sb1;
                unpack_f32x2(acc_a, sa0, sa1); unpack_f32x2(acc_b, sb0, sb1);
                const float sa = sa0 + sa1, sb = sb0 + sb1;
                if (renew || !__any_sync(0xffffffffu, fmaxf(sa, sb) > SUM_LIMIT)) { l_a += sa; l_b += sb; break; }
                renew = true;
            }
            if (!ok) break;
            // P goes over the scores it was computed from (this warp's own lanes, already in registers)
            tmem_st_16x128b_x8(t_tile + C::COL_SP + s * C::SP_STRIDE, pk);
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.p_ready[s]));   // one arrival per warp
        }
        // From here on addresses come from copies that the compiler knows nothing of: it would form all of them ahead of
        // the loop above and keep them in registers that the loop needs.
        int elane = lane;
        uint32_t sb = s_base;
        asm volatile("" : "+r"(elane), "+r"(sb));
        const int q4 = elane & 3, ra = lane0 + (elane >> 2), rb = ra + 8;
        float coef_a = 0.f, coef_b = 0.f;
        if (ok && linear) {
            // ReLU of the Q rows in place, and the denominators ReLU(Q_n) . Z: the four threads of a
            // row take two 16-byte groups of every 64 channels each.  Every Q K^T of this tile has
            // completed (its scores were consumed above), so Q is no longer read; the last P V
            // product may still be running meanwhile.
            // Rotary variant (Sec. 4.1): the numerator takes ReLU(Q) rotated pair by pair, the denominator
            // the un-rotated values.  A thread meets CH * 4 vectors of 8 channels; the (cos, sin) values of
            // each (16 bytes of the table, from L2) are fetched two vectors ahead, the first before the waits.
            constexpr int NIT = C::CH * 4;
            const bool rotary = p.rope != nullptr;
            auto rot_ptr = [&](int it) {
                const int row = (it & 1) ? rb : ra;
                const int tok = min(qb * p.Bq + row, p.N - 1);           // rows past the block or N hold zeros
                return reinterpret_cast<const uint4*>(p.rope + size_t(tok) * D + (it >> 2) * 64 +
                                                      (q4 + 4 * ((it >> 1) & 1)) * 8);
            };
            ok = wait_uniform(&bars.q_full, 0);
            if (ok) ok = wait_uniform(&bars.z_full, 0);
            if (ok) {
                // Four vectors are read before the first is written over (in turn, each load would wait for the store before it,
                // which may go to the same place for all the compiler knows), Z is read once for both rows, the rotary form
                // has a loop of its own: the pass takes 2000 cycles instead of 2700 at 12 heads of 32760 tokens.
                const uint32_t qa = sb + C::OFF_Q + ra * 128, sw_a = ra & 7;      // row b: 8 rows on, the same swizzle
                float den_a = 0.f, den_b = 0.f;
                auto pass = [&](auto with_rotation) {
                    constexpr bool ROT = decltype(with_rotation)::value;
                    uint4 tw[2];
                    if (ROT) { tw[0] = __ldg(rot_ptr(0)); tw[1] = __ldg(rot_ptr(1)); }
#pragma unroll
                    for (int ch = 0; ch < C::CH; ++ch) {
                        uint4 v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) v[u] = lds_128(qa + ch * C::Q_CHUNK + (u & 1) * 1024 + (((q4 + 4 * (u >> 1)) ^ sw_a) << 4));
#pragma unroll
                        for (int u2 = 0; u2 < 2; ++u2) {
                            const float4* zp = reinterpret_cast<const float4*>(z_s + ch * 64 + (q4 + 4 * u2) * 8);
                            const float4 z0 = zp[0], z1 = zp[1];                 // for both rows
                            const float z[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
#pragma unroll
                            for (int e2 = 0; e2 < 2; ++e2) {
                                const int u = u2 * 2 + e2, it = ch * 4 + u;
                                __nv_bfloat162* hv = reinterpret_cast<__nv_bfloat162*>(&v[u]);
                                const uint4 tv = ROT ? tw[u & 1] : make_uint4(0, 0, 0, 0);
                                if (ROT && it + 2 < NIT) tw[u & 1] = __ldg(rot_ptr(it + 2));
                                const __half2* th = reinterpret_cast<const __half2*>(&tv);      // (cos, sin) of four pairs
                                float den = 0.f;
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    hv[e] = __hmax2(hv[e], __float2bfloat162_rn(0.f));
                                    const float2 f = __bfloat1622float2(hv[e]);
                                    den = fmaf(f.x, z[2 * e], den);
                                    den = fmaf(f.y, z[2 * e + 1], den);
                                    if (ROT) {
                                        const float2 cs = __half22float2(th[e]);
                                        hv[e] = __floats2bfloat162_rn(cs.x * f.x - cs.y * f.y, cs.y * f.x + cs.x * f.y);
                                    }
                                }
                                if (e2) den_b += den; else den_a += den;
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) sts_128(qa + ch * C::Q_CHUNK + (u & 1) * 1024 + (((q4 + 4 * (u >> 1)) ^ sw_a) << 4), v[u]);
                    }
                };
                if (rotary) pass(std::true_type{}); else pass(std::false_type{});
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.lin_ready));
                den_a = quad_sum(den_a); den_b = quad_sum(den_b);
                // a row with ReLU(Q_n) = 0 and eps = 0 is 0/0: defined as 0 (the numerator is 0 as well)
                const float da = den_a + p.eps, db = den_b + p.eps;
                coef_a = da > 0.f ? item.scale / da : 0.f;
                coef_b = db > 0.f ? item.scale / db : 0.f;
            }
        }
        if (ok && len > 0) {
            ok = wait_uniform(&bars.o_final, 0);
            tc_fence_after_sync();
        }
        if (ok && linear) {
            ok = wait_uniform(&bars.lin_done, 0);
            tc_fence_after_sync();
        }

        if (ok) {
            // O = O_acc / l + coef * num, rounded once to bf16, staged over the V ring
            const float lt_a = quad_sum(l_a), lt_b = quad_sum(l_b);
            const float inv_a = (len > 0) ? 1.0f / lt_a : 0.f, inv_b = (len > 0) ? 1.0f / lt_b : 0.f;
#pragma unroll
            for (int cc = 0; cc < D / 32; ++cc) {
                uint32_t orr[16], nr[16];
                if (len > 0 && linear) tmem_ld_16x256b_x4(t_tile + C::COL_O + cc * 32, orr, t_tile + cc * 32, nr);
                else if (len > 0) tmem_ld_16x256b_x4(t_tile + C::COL_O + cc * 32, orr);
                else if (linear) tmem_ld_16x256b_x4(t_tile + cc * 32, nr);
                const uint32_t oa = sb + C::OFF_V + (cc >> 1) * C::Q_CHUNK + ra * 128 + q4 * 4;        // over the V ring
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f;
                    if (len > 0) {
                        a0 = __uint_as_float(orr[4 * n]) * inv_a;     a1 = __uint_as_float(orr[4 * n + 1]) * inv_a;
                        b0 = __uint_as_float(orr[4 * n + 2]) * inv_b; b1 = __uint_as_float(orr[4 * n + 3]) * inv_b;
                    }
                    if (linear) {
                        a0 = fmaf(coef_a, __uint_as_float(nr[4 * n]), a0);     a1 = fmaf(coef_a, __uint_as_float(nr[4 * n + 1]), a1);
                        b0 = fmaf(coef_b, __uint_as_float(nr[4 * n + 2]), b0); b1 = fmaf(coef_b, __uint_as_float(nr[4 * n + 3]), b1);
                    }
                    const int off = ((((cc & 1) * 4 + n) ^ (ra & 7)) << 4);       // 16-byte group (8 columns) within the row
                    sts_32(oa + off, pack_bf16x2(a0, a1));
                    sts_32(oa + 8 * 128 + off, pack_bf16x2(b0, b1));
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.out_staged));
            if (p.lse != nullptr && q4 == 0) {
#pragma unroll
                for (int e2 = 0; e2 < 2; ++e2) {
                    const int row = e2 ? rb : ra;
                    int n = qb * p.Bq + row;
                    if (perm) {                      // row = position within the block * T + frame
                        const int sp = qb * p.th.kq + row / p.th.T;
                        n = (sp < p.th.S) ? (row % p.th.T) * p.th.S + sp : p.N;
                    }
                    if (row < q_rows && n < p.N)
                        p.lse[size_t(bh) * p.N + n] =
                            (len > 0) ? ((e2 ? m_b : m_a) + log2f(e2 ? lt_b : lt_a)) * 0.6931471805599453f : -INFINITY;
                }
            }
        }
        }  // rows of queries
    }
    }  // !inherited_abort

    // ------------------------------------------------------------------ tear-down
    tc_fence_before_sync();
    __syncthreads();
    // The first kernel of the next call waits for this grid and for nothing before it, so this grid must not end ahead of the
    // state kernels of its own call, also where no CTA needed them (rejected lists, dropped items).
    // (Only there: the instruction is not free, 2 us of a 32 us call when every CTA issues it once more.)
    if ((p.mode & MODE_LINEAR) != 0 && (!linear || inherited_abort)) grid_dependency_wait();
    if (abort_flag != 0 && !inherited_abort) {
        // a bounded wait expired somewhere (1: in this CTA, reported here; 2: in the state kernels, which
        // reported it themselves): give copies in flight time to land, leave
        if (tid == 0 && abort_flag == 1) {
            atomicExch(p.ws_status, SALAD_ERR_TIMEOUT);
            if (p.user_status) atomicExch(p.user_status, SALAD_ERR_TIMEOUT);
        }
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 200000ull) { __nanosleep(1000); }
        __syncthreads();
    }
    if (warp == 2) tmem_dealloc(tmem, C::TMEM_COLS);
}

}  // namespace salad
