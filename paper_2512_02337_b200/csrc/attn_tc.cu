// Tensor-core verification attention for B200 (sm_100a): bfloat16, head_dim 64 or 128, pages of 16, 32 or 64 tokens.
// Tree-masked GQA attention of the step's tokens over a paged cache (paper Section 3.2-3.3,
// Algorithm 1 "TreeDecode"), used for both the partial and the full cache.
//
// One CTA owns one (layer, sequence, KV head, KV split, row group).  All G query heads of the KV head times
// floor(128/G) step tokens are packed into a 128-row tile, so QK^T and PV are dense 128x128xd and 128xdx128
// contractions.  Two streams of tiles run through the CTA in ping-pong, so that the contractions of one hide behind
// the softmax of the other:
//   two row tiles   stream t is row tile t; both streams walk the same K/V tiles
//   one row tile    stream t takes every other K/V tile of the one row tile, each stream with its own running maximum,
//                   sum and accumulator; the two are combined at the end.  (One stream alone leaves the tensor
//                   pipe idle during its softmax: 64K tokens x 36 layers, 32 query rows per head, 1715 -> 1457 us = the
//                   copy rate.)
//   warp 0      TMA producer: Q once, then K and V tiles of 128 tokens (2, 4 or 8 pages, one copy per page,
//               each issued by its own lane) through the block table into a ring of shared-memory slots
//               (128-byte swizzle)
//   warp 1      MMA issuer: tcgen05.mma  S_t = Q_t K^T  (both operands in shared memory) and
//               O_t += P_t V (P read from tensor memory, V MN-major from shared memory)
//   warps 4-7   softmax of stream 0, warps 8-11 of stream 1: one thread per row reads S from
//               tensor memory, keeps the running max / sum of an online softmax in the log2
//               domain, writes P (bfloat16) over S, rescales O only when the max grew by > 2^8,
//               and finally normalises O and writes it out
// Tensor memory (512 columns): S0 | S1 | O0 | O1, 128 columns each, P_t aliases S_t.
// With several KV splits the unnormalised (O, m, l) go to the workspace and merge_kernel combines
// them by log-sum-exp.  Every wait is bounded; a wait that gives up records SPECPV_ERR_TIMEOUT.
//
// Precision of the weights.  With 128 channels and a group size that divides 128, P is rounded to bfloat16 once.  Head size 64 and the
// other group sizes (kSplit) keep the float32 weights and accurate log-sum-exps of the plain kernel: P goes to the tensor core as two
// bfloat16 terms, the weight's upper half and what that leaves out, side by side over S (64 + 64 columns), the row sum is taken
// over the float32 weights, and the scale carries a second term (see scale_log2_lo).  Relative 2-norm errors against float64, one
// bfloat16 term / two / plain kernel: log-sum-exp 4.8e-5 / 3.5e-8 / 4.0e-8, bfloat16 output 1.86e-3 / 1.66e-3 / 1.66e-3 (1.66e-3 is its own
// rounding), float32 output 8.5e-4 / 5.5e-6 / 6.6e-7 (12345 tokens, 48 x 5 rows of 128; what is left is the tensor core
// cutting off the sums over the tokens), 5.4e-5 / 3.3e-8 / 3.4e-8, 1.79e-3 / 1.66e-3 / 1.66e-3 and 6.5e-4 / 4.5e-6 / 3.9e-7
// (4101 tokens, 60 x 4 rows of 64).  It takes half again the contractions of P V and a third more of the softmax: 24.6 -> 31.4 us and
// 16.1 -> 18.7 us for one layer, where the plain kernel took 1310 and 375.
#include "attn_tc.cuh"

namespace specpv {

namespace {

constexpr int kThreadsTc = 384;          // 12 warps

// Shared memory by head size: a Q tile is [d/64 parts][128 rows][64 d] bf16, a K or V tile [16 groups of 8 tokens][d/64 parts]
// [8 tokens][64 d], so that a page is contiguous and arrives in ONE copy of all its channels (a tensor map with the tokens
// split into groups of eight).  (The copy engine spends some 60 ns per box whatever it carries, and a copy per page and part
// made 16-token pages wait for it: 61440 tokens x 16 layers, 32 rows,
// 834 -> 675 us; a copy of half a page or a quarter is no faster.)
template <int D>
struct Shape {
    static constexpr int kParts = D / 64;
    static constexpr int kSlotBytes = kTileTokens * D * 2;
    static constexpr int kStages = D == 128 ? 5 : 10;
    static constexpr int kGroupBytes = 8 * D * 2;  // eight tokens of a K or V tile
    static constexpr int kQTileBytes = 128 * D * 2;
    static constexpr int kQBytes = 2 * kQTileBytes;
    static constexpr int kSmemBytes = 1024 + kQBytes + kStages * kSlotBytes;
};
constexpr int kMaxStages = 10;
constexpr int kShortWalk = 4;  // tiles per CTA

using namespace tc;

// Instruction descriptors, kind::f16: accumulator f32, A = B = bf16, M = 128, N = 128 tokens (QK) or D channels (PV).
constexpr uint32_t kIdescQK = make_idesc(128, false);
template <int D>
constexpr uint32_t kIdescPV = make_idesc(D, true);  // B (= V) is MN-major

struct __align__(8) Barriers {
    uint64_t q_full;
    uint64_t kv_full[kMaxStages];   // a K or V tile has landed in its slot
    uint64_t kv_empty[kMaxStages];  // every contraction that reads the slot has completed (one barrier per slot: a barrier
                                    // shared by all slots could run two phases ahead of the producer, which a parity
                                    // wait cannot tell from none)
    uint64_t s_full[2];         // phase j: the j-th S of stream t is complete
    uint64_t p_full[2];         // phase j: the four softmax warps of stream t have stored their j-th P
    uint64_t o_done[2];         // the last PV of stream t has completed
    uint64_t v_need;            // MMA issuer -> warp 2: this V tile has landed and needs its tail rows zeroed
    uint64_t v_fixed;           // warp 2 -> MMA issuer: done
    uint64_t drain;             // completion of the contractions issued before a wait gave up
    uint32_t tmem_base;
    int abort_flag;
};

// What every role of a CTA knows about its work.
struct Job {
    uint8_t* smem;
    uint32_t q_smem, tmem;
    int split, rg, h, lb, b, l;
    int seq_len, M, tok_per_tile, tile_rows, tok0;
    int tile_begin, n_ctx_tiles, n_tiles, first_fix;
};

// The roles.  kOne: the row group is one row tile and the streams take alternate K/V tiles.
// K/V tiles go through the ring in the order in which the issuer releases them: V(i - lag), then K(i), where lag is the
// number of S buffers that a row tile has (two row tiles: one each, lag 1; one row tile: both, lag 2).

// =========================== TMA producer ================================================
template <int D>
__device__ __forceinline__ void copy_q(const TcParams& p, const Job& c, Barriers& bars, bool one, int lane) {
    using Sh = Shape<D>;
    const uint32_t qbar = smem_u32(&bars.q_full);
    const int n_q_tiles = one ? 1 : 2;
    if (lane == 0) {
        mbar_expect_tx(qbar, (uint32_t)(n_q_tiles * Sh::kParts * c.tile_rows * 128));
        for (int t = 0; t < n_q_tiles; ++t)
            for (int part = 0; part < Sh::kParts; ++part)
                tma_load_4d(c.q_smem + t * Sh::kQTileBytes + part * 16384, &p.tm_q, part * 64, c.h * p.G,
                            c.tok0 + t * c.tok_per_tile, c.lb, qbar);
    }
    __syncwarp();
}

// Pool group coordinate (eight tokens each) of page `lane` of context tile j (128 / page size of them).  The lane that looks
// a page up later issues its copy, so that a tile's copies leave in one pass of the warp; the table is read one tile
// ahead so that its latency hides behind the wait for a free slot.
__device__ __forceinline__ int page_group(const TcParams& p, const Job& c, int j, int lane) {
    const int ppt = kTileTokens / p.bs;
    int group = (int)(p.pool_rows / 8);  // out of range: the copy engine fills zeros
    const int blk = (c.tile_begin + j) * ppt + lane;
    if (lane < ppt && j < c.n_ctx_tiles && (long long)blk * p.bs < c.seq_len && blk < p.max_blocks) {
        const int page = p.block_table[(size_t)c.b * p.max_blocks + blk];
        if (page < 0 || page >= p.n_pages)
            record_fault(p.workspace, SPECPV_ERR_BAD_BLOCK_TABLE, c.b, blk, page, c.l);
        else
            group = (int)((((long long)(p.layer0 + c.l) * p.n_pages + page) * p.Hkv + c.h) * (p.bs / 8));
    }
    return group;
}

// The whole warp runs the loop (a lone lane of a diverged warp runs slowly).
template <int D>
__device__ __forceinline__ void produce(const TcParams& p, const Job& c, Barriers& bars, bool one, int lane) {
    using Sh = Shape<D>;
    constexpr int kStages = Sh::kStages, kParts = Sh::kParts, kSlotBytes = Sh::kSlotBytes;
    const int lag = one ? 2 : 1;
    volatile int* abort_flag = &bars.abort_flag;
    const uint32_t kv_smem = c.q_smem + Sh::kQBytes;
    const int ppt = kTileTokens / p.bs;
    const uint32_t page_off = lane * (p.bs / 8) * Sh::kGroupBytes;
    const int new_groups = (c.M + 7) / 8;  // groups of the step's own tokens
    bool ok = true;
    int at_k = 0, at_v1 = 0, at_v2 = 0, at_next = page_group(p, c, 0, lane);  // of tiles i, i - 1, i - 2, i + 1
    uint32_t slot = 0, par = 1, use = 0;  // ring position of the next use; parity of the release that frees its slot
    for (int i = 0; i < c.n_tiles + lag; ++i) {
        at_v2 = at_v1;
        at_v1 = at_k;
        at_k = at_next;
        at_next = page_group(p, c, i + 1, lane);
        for (int kv = 1; kv >= 0; --kv) {  // 1: V tile, 0: K tile
            const int j = kv ? i - lag : i;
            if (j < 0 || j >= c.n_tiles) continue;
            const uint32_t full = smem_u32(&bars.kv_full[slot]), empty = smem_u32(&bars.kv_empty[slot]);
            // After a wait that gave up nothing more is copied.  The lanes leave each by itself, and meet nowhere in these loops: a vote ahead of
            // the copies makes short calls 0.5 % slower, one behind them those with 16-token pages 1 %.
            if (use >= (uint32_t)kStages) ok = mbar_wait(empty, par, abort_flag, p.workspace, 1);
            if (!ok) break;  // each lane by itself
            const uint32_t dst = kv_smem + slot * kSlotBytes;
            if (j >= c.n_ctx_tiles) {  // the step's own tokens, a copy per group and part; the rest of the slot is masked or zeroed
                if (lane == 0) mbar_expect_tx(full, new_groups * Sh::kGroupBytes);
                if (lane < new_groups * kParts)
                    tma_load_3d(dst + lane * 1024, kv ? &p.tm_vnew : &p.tm_knew, lane % kParts * 64, c.h,
                                c.lb * p.M_max + lane / kParts * 8, full);
            } else {
                if (lane == 0) mbar_expect_tx(full, kSlotBytes);
                if (lane < ppt)
                    tma_load_4d(dst + page_off, kv ? &p.tm_vpool : &p.tm_kpool, 0, 0, 0, kv ? (one ? at_v2 : at_v1) : at_k, full);
            }
            ++use;
            if (++slot == kStages) { slot = 0; par ^= 1; }
        }
        if (!ok) break;  // each lane by itself
    }
}

// =========================== MMA issuer ==================================================
// One warp issues every contraction (issuing from two warps serialises the tensor pipe).  Issue
// order (ping-pong of the two streams): QK(0,0) QK(0,1) | PV(0,0) QK(1,0) PV(0,1) QK(1,1) | ...
// Barrier instructions do not overlap with queued MMAs (each costs the pipe 30-100 idle cycles),
// so the loop keeps them to four waits per KV tile, without votes, and four commits behind MMAs.  The whole
// warp runs the loop, lane 0 issues.
template <int D, bool kOne, bool kSplit>
__device__ __forceinline__ void issue(const TcParams& p, const Job& c, Barriers& bars, int lane) {
    using Sh = Shape<D>;
    constexpr int kStages = Sh::kStages;
    constexpr uint32_t kSlotWords = Sh::kSlotBytes >> 4, kQTileWords = Sh::kQTileBytes >> 4;  // 16-byte units of descriptors
    volatile int* abort_flag = &bars.abort_flag;
    const uint32_t kv_smem = c.q_smem + Sh::kQBytes, tmem = c.tmem;
    const int n_tiles = c.n_tiles, first_fix = c.first_fix;
    bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.q_full), 0, abort_flag, p.workspace, 2));
    // Shared-memory descriptors: the upper word (stride between 8-row groups, version, swizzle) is
    // constant; the lower word is the 16-byte address plus the leading-dimension offset (V: to the next 64 channels).
    const uint32_t q_hi = (uint32_t)((1024u >> 4) | (1u << 14) | (2u << 29));
    const uint32_t kv_hi = (uint32_t)((Sh::kGroupBytes >> 4) | (1u << 14) | (2u << 29));
    const uint32_t q_lo = ((c.q_smem >> 4) & 0x3FFFu) | ((16u >> 4) << 16);
    const uint32_t k_lo0 = ((kv_smem >> 4) & 0x3FFFu) | ((16u >> 4) << 16);
    const uint32_t v_lo0 = ((kv_smem >> 4) & 0x3FFFu) | ((1024u >> 4) << 16);
    const uint32_t full0 = smem_u32(&bars.kv_full[0]), empty0 = smem_u32(&bars.kv_empty[0]);
    const uint32_t sfull0 = smem_u32(&bars.s_full[0]), pfull0 = smem_u32(&bars.p_full[0]);
    auto issue_pv = [&](int t, uint32_t vb_lo, bool first) {  // O_t (+)= P_t V
        const uint32_t a = tmem + t * 128, d = tmem + 256 + t * 128;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {  // 16 tokens per instruction: two groups
            const uint32_t b = vb_lo + (uint32_t)kk * (2 * Sh::kGroupBytes >> 4);
            mma_ts_lohi(d, a + kk * 8, b, kv_hi, kIdescPV<D>, (!first || kk > 0) ? 1u : 0u);
            if (kSplit) mma_ts_lohi(d, a + 64 + kk * 8, b, kv_hi, kIdescPV<D>, 1u);
        }
    };
    auto issue_qk = [&](int t, uint32_t a_lo, uint32_t kb_lo) {  // S_t = Q K^T
        const uint32_t d = tmem + t * 128;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {  // 16 channels per instruction
            const uint32_t q_off = (uint32_t)((kk >> 2) * 16384 + (kk & 3) * 32) >> 4, k_off = (uint32_t)((kk >> 2) * 1024 + (kk & 3) * 32) >> 4;
            mma_ss_lohi(d, a_lo + q_off, q_hi, kb_lo + k_off, kv_hi, kIdescQK, kk > 0 ? 1u : 0u);
        }
    };
    // Ring uses: K0 | V0 K1 | V1 K2 | .. with two row tiles, K0 | K1 | V0 K2 | V1 K3 | .. with one.
    // A wait that gives up raises the abort flag, which makes the later waits of this tile return at once; the
    // loop ends after this tile, so at most one tile's contractions are issued past the failed wait.  (One exit
    // per tile: an exit after every wait costs the issuing thread 7 % of the kernel.)  The lanes leave together, on a vote: they
    // test the barrier and the flag each for itself, and one that left alone would be missing where the others meet.
    if (!kOne) {
        uint32_t k_slot = 0, k_par = 0, v_slot = 1, v_par = 0;  // slot and phase parity of the next K and V tile
        for (int j = 0; j <= n_tiles; ++j) {
            const int jp = j - 1;
            if (j < n_tiles) ok &= mbar_wait(full0 + k_slot * 8, k_par, abort_flag, p.workspace, 3);
            if (j > 0) {
                ok &= mbar_wait(full0 + v_slot * 8, v_par, abort_flag, p.workspace, 4);
                // a ragged or tree tile: warp 2 zeroes the rows of V past the valid tokens first
                if (jp >= first_fix) {
                    if (lane == 0) mbar_arrive(smem_u32(&bars.v_need));
                    ok &= mbar_wait(smem_u32(&bars.v_fixed), (jp - first_fix) & 1, abort_flag, p.workspace, 9);
                }
            }
            const uint32_t kb_lo = launder(k_lo0 + k_slot * kSlotWords);
            const uint32_t vb_lo = launder(v_lo0 + v_slot * kSlotWords);
            for (int t = 0; t < 2; ++t) {
                if (j > 0) {
                    ok &= mbar_wait(pfull0 + t * 8, jp & 1, abort_flag, p.workspace, 5);
                    tc_fence_after();
                }
                if (lane == 0) {
                    if (j > 0) {
                        issue_pv(t, vb_lo, jp == 0);
                        if (t == 1) tc_commit(empty0 + v_slot * 8);
                        if (j == n_tiles) tc_commit(smem_u32(&bars.o_done[t]));
                    }
                    if (j < n_tiles) {
                        issue_qk(t, launder(q_lo + (uint32_t)t * kQTileWords), kb_lo);
                        tc_commit(sfull0 + t * 8);
                        if (t == 1) tc_commit(empty0 + k_slot * 8);
                    }
                }
                if (t == 0) __syncwarp();
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (j < n_tiles) { k_slot += 2; if (k_slot >= kStages) { k_slot -= kStages; k_par ^= 1; } }
            if (j > 0) { v_slot += 2; if (v_slot >= kStages) { v_slot -= kStages; v_par ^= 1; } }
        }
    } else {
        uint32_t slot = 0, par = 0;
        auto advance = [&] { if (++slot == kStages) { slot = 0; par ^= 1; } };
        for (int i = 0; i < n_tiles + 2; ++i) {
            const int t = i & 1, jv = i - 2;
            uint32_t k_slot = 0, v_slot = 0;
            if (jv >= 0) {
                v_slot = slot;
                ok &= mbar_wait(full0 + slot * 8, par, abort_flag, p.workspace, 4);
                advance();
                if (jv >= first_fix) {
                    if (lane == 0) mbar_arrive(smem_u32(&bars.v_need));
                    ok &= mbar_wait(smem_u32(&bars.v_fixed), (jv - first_fix) & 1, abort_flag, p.workspace, 9);
                }
                ok &= mbar_wait(pfull0 + t * 8, (jv >> 1) & 1, abort_flag, p.workspace, 5);
            }
            if (i < n_tiles) {
                k_slot = slot;
                ok &= mbar_wait(full0 + slot * 8, par, abort_flag, p.workspace, 3);
                advance();
            }
            tc_fence_after();
            if (lane == 0) {
                if (jv >= 0) {
                    issue_pv(t, launder(v_lo0 + v_slot * kSlotWords), jv < 2);
                    tc_commit(empty0 + v_slot * 8);
                    if (i >= n_tiles) tc_commit(smem_u32(&bars.o_done[t]));
                }
                if (i < n_tiles) {
                    issue_qk(t, q_lo, launder(k_lo0 + k_slot * kSlotWords));
                    tc_commit(sfull0 + t * 8);
                    tc_commit(empty0 + k_slot * 8);
                }
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
        }
    }
    if (!ok && lane == 0) {
        // after a give-up: wait (bounded) until the contractions that WERE issued have completed, so that the
        // tensor memory is not freed under them
        tc_commit(smem_u32(&bars.drain));
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(smem_u32(&bars.drain), 0) && global_ns() - t0 < 100000000ull) {}
    }
    __syncwarp();
}

// =========================== V fixer =====================================================
// Rows of a V tile past its valid tokens may hold anything (stale shared memory, rows of other
// sequences' steps): zero them so that 0 * garbage cannot produce NaN.  Only the last context
// tile (when ragged) and the tile of the step's own tokens can need it.
template <int D, bool kOne>
__device__ __forceinline__ void fix_v(const TcParams& p, const Job& c, Barriers& bars, int lane) {
    using Sh = Shape<D>;
    for (int jp = c.first_fix; jp < c.n_tiles; ++jp) {
        const int use = kOne && jp < c.n_tiles - 1 ? 2 * jp + 2 : 2 * jp + 1;  // the ring use of V(jp)
        // the request arrives once the tile has landed (a wait on the slot's own barrier this far
        // ahead of the pipeline could match an earlier phase of the same parity)
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.v_need), (jp - c.first_fix) & 1, &bars.abort_flag, p.workspace, 10)))
            break;
        const int n_valid = jp >= c.n_ctx_tiles ? c.M : min(kTileTokens, c.seq_len - (c.tile_begin + jp) * kTileTokens);
        uint8_t* v = c.smem + Sh::kQBytes + (size_t)(use % Sh::kStages) * Sh::kSlotBytes;
        // a lane keeps its 16-byte column, the warp takes 32 / (8 kParts) rows at a time (the last split of a short call
        // waits for this: with the row and column worked out per store it took a microsecond longer)
        constexpr int kRowsAtOnce = 32 / (8 * Sh::kParts);
        v += lane / 8 % Sh::kParts * 1024 + lane % 8 * 16;
#pragma unroll 4
        for (int r = n_valid + lane / (8 * Sh::kParts); r < kTileTokens; r += kRowsAtOnce)
            *reinterpret_cast<uint4*>(v + (r >> 3) * Sh::kGroupBytes + (r & 7) * 128) = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.v_fixed));
    }
}

// =========================== softmax / correction / epilogue ==============================
// A warp none of whose rows is in use (38 tokens x 4 heads leave three of the eight without) passes zeros on, and leaves the
// exponentials to the warp that shares its scheduler and the power to the rest: 64K tokens x 36 layers, 38 rows per head
// 2080 -> 1956 us, 48 rows 2080 -> 2005, 13 rows 1378 -> 1320; 60 rows, which use every warp, 2080 either way.
template <bool kSplit>
__device__ __noinline__ void pass_zeros(const TcParams& p, Barriers& bars, int t, int first_tile, int step, int n_tiles,
                                        uint32_t s_addr, int lane) {
    volatile int* abort_flag = &bars.abort_flag;
    uint32_t zero[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) zero[i] = 0;
    uint32_t s_par = 0;
    bool ok = true;
    for (int j = first_tile; j < n_tiles; j += step, s_par ^= 1) {
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.s_full[t]), s_par, abort_flag, p.workspace, 6));
        if (!ok) return;
        tc_fence_after();
        TMEM_ST32(s_addr, zero);
        TMEM_ST32(s_addr + 32, zero);
        if (kSplit) {
            TMEM_ST32(s_addr + 64, zero);
            TMEM_ST32(s_addr + 96, zero);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.p_full[t]));
    }
    mbar_wait(smem_u32(&bars.o_done[t]), 0, abort_flag, p.workspace, 8);  // its contractions have ended before the CTA does
}

template <int D, bool kOne, bool kSplit>
__device__ __forceinline__ void softmax(const TcParams& p, const Job& c, Barriers& bars, int warp, int lane) {
    using Sh = Shape<D>;
    volatile int* abort_flag = &bars.abort_flag;
    const int t = (warp - 4) >> 2;           // stream of this warpgroup
    const int q = warp & 3;                  // TMEM lane quarter this warp may access
    const int row_in_tile = q * 32 + lane;
    const int n_tiles = c.n_tiles;
    constexpr int step = kOne ? 2 : 1;
    const int first_tile = kOne ? t : 0;     // K/V tiles of this stream: first_tile, first_tile + step, ..
    // (two row tiles: n_tiles is never 0 here; said, it changes the loop's code, 33 rows x 4 of 64 channels, 16000 tokens x 6
    // layers 99.7 -> 98.2 us)
    if (!kOne && n_tiles <= 0) return;
    const bool idle = kOne && first_tile >= n_tiles;  // one tile: nothing for stream 1, which still does the dry run below
    const int row_tile = kOne ? 0 : t;
    const int row = row_tile * 128 + row_in_tile;                              // row within the row group
    const int tok = c.tok0 + row_tile * c.tok_per_tile + row_in_tile / p.G;    // step token of this row
    const int g = row_in_tile % p.G;
    const bool row_valid = row_in_tile < c.tile_rows && tok < c.M;
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const uint32_t s_addr = c.tmem + lane_addr + t * 128;
    const uint32_t o_addr = c.tmem + lane_addr + 256 + t * 128;
    if (!__any_sync(0xffffffffu, row_valid)) {
        if (idle) return;
        pass_zeros<kSplit>(p, bars, t, first_tile, step, n_tiles, s_addr, lane);
        if (kOne && n_tiles > 1) asm volatile("bar.sync 1, 256;" ::: "memory");  // where the two streams meet below
        return;
    }
    uint64_t mask_lo = 0, mask_hi = 0;
    if (row_valid) {
        const uint64_t* mrow = p.tree_mask + ((size_t)c.b * p.M_max + tok) * p.mask_words;
        mask_lo = mrow[0];
        if (p.mask_words > 1) mask_hi = mrow[1];
    }
    float m_run = -INFINITY, l_run = 0.f;
    bool ok = true;
    const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), sc2_lo = make_float2(p.scale_log2_lo, p.scale_log2_lo);
    // One row tile (the form of short calls): the first pass of the loop is a dry run over zeros by stream 1, whose S comes
    // last or not at all, while Q and the first K tile are still on their way: it brings the loop's code (straight-line) into
    // the instruction cache.  In a model's layer other kernels have run since the last call, and with cold code the first
    // tile took 4.6-5 us from S to P instead of 1.5.  It passes through what a stream's first tile needs, the general path: through
    // both paths, and by stream 0 in CTAs of one tile, whose S then waited for it, it took twice as long (us per layer: 8 rows x 4,
    // 1024 tokens 10.5 -> 9.6; 26 rows x 4 of 64 channels, 1500 and 811 tokens 14.0 -> 13.4; 48 rows x 5, 12345 tokens
    // 32.0 -> 30.4).  (The form with two row tiles walks long contexts, where its loop ran 8 % slower with the dry run in it.)
    const bool warm_up = kOne && t == 1;
    uint32_t s_par = warm_up ? 1 : 0;
    for (int j = warm_up ? first_tile - step : first_tile; j < n_tiles && ok; j += step, s_par ^= 1) {
        const bool dry = kOne && j < first_tile;
        const bool is_new = j >= c.n_ctx_tiles;
        const int n_valid = is_new ? c.M : min(kTileTokens, c.seq_len - (c.tile_begin + j) * kTileTokens);
        const bool masked = is_new || n_valid < kTileTokens;
        uint64_t vis_lo = ~0ull, vis_hi = ~0ull;  // visibility of the tile's 128 columns for this row
        if (masked) {
            if (is_new) {
                vis_lo = mask_lo;
                vis_hi = mask_hi;
            }
            if (n_valid < 64) {
                vis_lo &= (n_valid <= 0) ? 0ull : (~0ull >> (64 - n_valid));
                vis_hi = 0;
            } else if (n_valid < 128) {
                vis_hi &= (n_valid == 64) ? 0ull : (~0ull >> (128 - n_valid));
            }
        }
        // the whole row of S (128 columns) goes to registers in one round trip
        uint32_t v[128];
        auto load_s = [&] {
            TMEM_LD32(s_addr, v);
            TMEM_LD32(s_addr + 32, (v + 32));
            TMEM_LD32(s_addr + 64, (v + 64));
            TMEM_LD32(s_addr + 96, (v + 96));
            tmem_wait_ld();
        };
        if (!dry) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.s_full[t]), s_par, abort_flag, p.workspace, 6));
            if (!ok) break;
            tc_fence_after();
            load_s();
        } else {
#pragma unroll
            for (int i = 0; i < 128; ++i) v[i] = 0;
        }
        // P = 2^(s*scale - m) as bf16 pairs, packed in place: word i of P (columns 2i, 2i+1) overwrites
        // v[i], whose own value was consumed by an earlier pair, so no second register array is needed.
        // The row sum is taken over the ROUNDED weights the tensor core will use, so that O / l is an
        // exact weighted average of V rows (the rounding error of a dominant weight cancels instead of
        // scaling the output).  kSplit: over the float32 weights, which the two terms hold to 2^-16.
        // kSplit: the first term is the weight cut to its upper half, the second what that took off, as bf16 pairs.  Neither term of a
        // weight is ever negative or zero (the second has 2^-23 of the weight added), so that a weight times an infinite
        // value stays infinite.
        constexpr float kOnePlus = 1.f + 1.1920929e-7f;
        uint32_t rest[kSplit ? 64 : 1];
        auto exp_row = [&](float m_use) {
            const float2 nm2 = make_float2(-m_use, -m_use);
            float2 sum2[4];  // independent partial sums: one chain of 64 dependent adds would outlast the exponentials
#pragma unroll
            for (int e = 0; e < 4; ++e) sum2[e] = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 64; ++i) {
                const float2 sv = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
                float2 x = __ffma2_rn(sv, sc2, nm2);
                if constexpr (kSplit) x = __ffma2_rn(sv, sc2_lo, x);
                const float2 e = make_float2(ex2(x.x), ex2(x.y));
                if constexpr (kSplit) {
                    const uint32_t ex = __float_as_uint(e.x), ey = __float_as_uint(e.y);
                    v[i] = __byte_perm(ex, ey, 0x7632);  // the upper halves
                    const float2 minus_upper = make_float2(__uint_as_float((ex & 0xFFFF0000u) | 0x80000000u),
                                                           __uint_as_float((ey & 0xFFFF0000u) | 0x80000000u));
                    const float2 r = __ffma2_rn(e, make_float2(kOnePlus, kOnePlus), minus_upper);
                    rest[i] = pack_bf16(r.x, r.y);
                    sum2[i & 3] = __fadd2_rn(sum2[i & 3], e);
                } else {
                    const uint32_t w = pack_bf16(e.x, e.y);
                    v[i] = w;
                    add_bf16_pair(sum2[i & 3], w);
                }
            }
            const float2 s01 = __fadd2_rn(sum2[0], sum2[1]), s23 = __fadd2_rn(sum2[2], sum2[3]);
            return (s01.x + s23.x) + (s01.y + s23.y);
        };
        // Fast path (every full context tile after the stream's first): keep the reference m_run of the row as it
        // is and skip the row maximum.  Weights may then exceed 1; float32 sums and bf16 weights keep
        // their relative precision whatever the exponent, so only overflow has to be ruled out: if a
        // row sum leaves the safe range (or a row has no reference yet), the warp takes the tile again
        // from tensor memory on the general path, which brings m_run up to date.  A short walk of the two-term form, whose fast path
        // would be met with cold code, stays on the general path (40 rows x 4 of 64 channels, 4 tiles per CTA: 17.8 -> 17.3 us).
        float l_add = 0.f;
        bool general = (kOne ? j <= first_tile : j == first_tile) || masked || (kOne && kSplit && n_tiles <= kShortWalk);
        if (!general) {
            l_add = exp_row(m_run);
            const bool bad = !(l_add < kSafeRowSum) || m_run == -INFINITY;
            if (__any_sync(0xffffffffu, bad)) {
                general = true;
                load_s();  // S_t is still intact: P has not been stored yet
            }
        }
        if (general) {
            if (masked) {  // ragged or tree-masked tile: invisible columns become -inf (at most two tiles per CTA)
#pragma unroll
                for (int i = 0; i < 128; ++i) {
                    const uint64_t word = i < 64 ? vis_lo : vis_hi;
                    if (!((word >> (i & 63)) & 1ull)) v[i] = 0xff800000u;
                }
            }
            float mx0 = __uint_as_float(v[0]), mx1 = __uint_as_float(v[1]), mx2 = __uint_as_float(v[2]),
                  mx3 = __uint_as_float(v[3]);
#pragma unroll
            for (int i = 4; i < 124; i += 8) {  // three-input max: two new values per instruction
                mx0 = fmax3(mx0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
                mx1 = fmax3(mx1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
                mx2 = fmax3(mx2, __uint_as_float(v[i + 4]), __uint_as_float(v[i + 5]));
                mx3 = fmax3(mx3, __uint_as_float(v[i + 6]), __uint_as_float(v[i + 7]));
            }
            mx0 = fmax3(mx0, __uint_as_float(v[124]), __uint_as_float(v[125]));
            mx1 = fmax3(mx1, __uint_as_float(v[126]), __uint_as_float(v[127]));
            const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3));
            const float m_tile = mx * p.scale_log2;
            // lazy rescale: keep the old reference max unless the new one is more than 2^8 larger.
            // The decision is per row, the tensor-memory traffic is warp-wide: if any row of the
            // warp rescales, all 32 rows pass through it (with a factor of 1 where nothing changes).
            bool need = false;
            if (kOne ? j <= first_tile : j == first_tile) {
                m_run = m_tile;
            } else {
                need = m_tile > m_run + kRescaleThreshold || (m_run == -INFINITY && m_tile > -INFINITY);
            }
            if (__any_sync(0xffffffffu, need)) {
                const float factor = !need ? 1.f : (m_run == -INFINITY ? 0.f : ex2(m_run - m_tile));
                // O_t already holds every earlier PV of this stream: the tensor pipe runs in order, and S_t, issued
                // after them, is complete
#pragma unroll (kOne ? 1 : D / 32)
                for (int cc = 0; cc < D / 32; ++cc) {
                    uint32_t o[32];
                    TMEM_LD32(o_addr + cc * 32, o);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * factor);
                    TMEM_ST32(o_addr + cc * 32, o);
                }
                if (need) {
                    l_run *= factor;
                    m_run = m_tile;
                }
            }
            l_add = exp_row(m_run == -INFINITY ? 0.f : m_run);
        }
        if (dry) {
            l_run = l_add < 0.f ? l_add : 0.f;  // never negative: zero again, and the dry run's sums are not dead code
            if (idle) return;
            continue;
        }
        TMEM_ST32(s_addr, v);
        TMEM_ST32(s_addr + 32, (v + 32));
        if constexpr (kSplit) {
            TMEM_ST32(s_addr + 64, rest);
            TMEM_ST32(s_addr + 96, (rest + 32));
        }
        l_run += l_add;
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars.p_full[t]));
    }
    // ---- epilogue: wait for the last PV, normalise, write out ---------------------------
    // One row tile, both streams in use: stream t finishes channels [t D/2, (t+1) D/2) from both accumulators, which the warps of
    // either stream reach (a warp's tensor-memory lanes are those of its place in the warpgroup); only maxima and sums go through
    // shared memory.  (Through shared memory, half an accumulator each way: one layer, 60 rows x 4, 4096 tokens 16.7 us against
    // 15.8, 16384 tokens 27.5 against 26.5, 26 rows x 4 of 64 channels, 1500 and 811 tokens 13.4 against 12.8.)
    const bool meet = kOne && n_tiles > 1;
    constexpr int kHalfD = D / 2;
    float w_mine = 1.f, w_other = 0.f;  // weights of the two streams relative to their common maximum
    if (meet) {
        float* xml = reinterpret_cast<float*>(c.smem + Sh::kQTileBytes);  // [2][2][128]: reference maximum, row sum (no second Q tile here)
        xml[t * 256 + row_in_tile] = m_run;
        xml[t * 256 + 128 + row_in_tile] = l_run;
        __syncwarp();
        asm volatile("bar.sync 1, 256;" ::: "memory");  // both streams' warps come here, whatever their waits returned
        const float m_o = xml[(1 - t) * 256 + row_in_tile], l_o = xml[(1 - t) * 256 + 128 + row_in_tile];
        const float m_all = fmaxf(m_run, m_o);
        w_mine = m_run == -INFINITY ? 0.f : ex2(m_run - m_all);
        w_other = m_o == -INFINITY ? 0.f : ex2(m_o - m_all);
        l_run = l_run * w_mine + l_o * w_other;
        m_run = m_all;
        ok = __all_sync(0xffffffffu, ok && !*abort_flag);
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.o_done[1 - t]), 0, abort_flag, p.workspace, 8));
    }
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars.o_done[t]), 0, abort_flag, p.workspace, 8));
    if (!ok) return;
    tc_fence_after();
    const bool direct = p.n_splits == 1;
    const float inv = direct ? 1.f / l_run : 1.f;
    w_mine *= inv;
    w_other *= inv;
    const size_t out_row = ((size_t)c.lb * p.M_max + tok) * p.Hq + c.h * p.G + g;
    const size_t prow = (((size_t)c.lb * p.Hkv + c.h) * p.n_splits + c.split) * p.R_pad + c.rg * p.rg_tiles * 128 + row;
    const int c_begin = meet ? t * kHalfD : 0, c_end = meet ? c_begin + kHalfD : D;
#pragma unroll (kOne ? 1 : D / 32)
    for (int c0 = c_begin; c0 < c_end; c0 += 32) {
        uint32_t v[32];
        TMEM_LD32(o_addr + c0, v);
        if (meet) {
            uint32_t other[32];
            TMEM_LD32(c.tmem + lane_addr + 256 + (1 - t) * 128 + c0, other);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * w_mine + __uint_as_float(other[i]) * w_other);
        } else {
            tmem_wait_ld();
        }
        if (!row_valid) continue;
        if (!meet && direct) {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * inv);
        }
        if (!direct) {
            // a thread's row is contiguous: 32-byte stores fill whole sectors, half as many
            // memory transactions as 16-byte ones for this one-row-per-lane pattern
            float* dst = p.part_o + prow * D + c0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + 8 * i),
                             "r"(v[8 * i]), "r"(v[8 * i + 1]), "r"(v[8 * i + 2]), "r"(v[8 * i + 3]), "r"(v[8 * i + 4]),
                             "r"(v[8 * i + 5]), "r"(v[8 * i + 6]), "r"(v[8 * i + 7])
                             : "memory");
        } else if (p.out_f32) {  // the caller's buffer: 16-byte aligned
            uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<float*>(p.out) + out_row * D + c0);
#pragma unroll
            for (int i = 0; i < 8; ++i) dst[i] = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        } else {
            uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p.out) + out_row * D + c0);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint4 w;
                w.x = pack_bf16(__uint_as_float(v[8 * i]), __uint_as_float(v[8 * i + 1]));
                w.y = pack_bf16(__uint_as_float(v[8 * i + 2]), __uint_as_float(v[8 * i + 3]));
                w.z = pack_bf16(__uint_as_float(v[8 * i + 4]), __uint_as_float(v[8 * i + 5]));
                w.w = pack_bf16(__uint_as_float(v[8 * i + 6]), __uint_as_float(v[8 * i + 7]));
                dst[i] = w;
            }
        }
    }
    if (row_valid && (!meet || t == 0)) {
        if (direct) {
            if (p.lse) p.lse[out_row] = fmaf(m_run, kLn2, logf(l_run));
        } else {
            p.part_ml[prow * 2] = m_run;  // log2 units, unrounded: the merge takes differences of them
            p.part_ml[prow * 2 + 1] = l_run;
        }
    }
}

// =================================================================================================
// kSplit: P as two bfloat16 terms (head size 64 and group sizes that do not divide 128).
// kForm: the row groups a launch can meet (a kernel with both forms has twice the code, which a call that follows other
// kernels pays for in instruction-cache misses).
enum { kOneTile, kTwoTiles, kBoth };
template <int D, int kForm, bool kSplit>
__global__ void __launch_bounds__(kThreadsTc, 1) attn_tc_kernel(const __grid_constant__ TcParams p) {
    using Sh = Shape<D>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ Barriers bars;
    Job c;
    // 1024-byte alignment for the 128-byte swizzle atoms
    c.smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // CTA order: all full row groups first (those of a head side by side, they read the same K/V), then the row groups of
    // one tile, which are shorter and fill the machine's tail
    c.split = blockIdx.x % p.n_splits;
    int unit = blockIdx.x / p.n_splits;
    if (unit < p.n_full_units) {
        c.rg = unit % p.n_full_groups;
        unit /= p.n_full_groups;
    } else {
        c.rg = p.n_full_groups;
        unit -= p.n_full_units;
    }
    c.h = unit % p.Hkv;
    c.lb = unit / p.Hkv;
    c.b = c.lb % p.batch;
    c.l = c.lb / p.batch;

    c.tok_per_tile = 128 / p.G;                  // step tokens per 128-row tile
    c.tile_rows = c.tok_per_tile * p.G;          // rows of a tile in use (all 128 when G divides 128)
    c.tok0 = c.rg * p.rg_tiles * c.tok_per_tile; // first step token of this row group

    // ---- set-up (nothing here depends on earlier work on the stream) ----------------------------
    c.q_smem = smem_u32(c.smem);
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&bars.q_full), 1);
        for (int s = 0; s < Sh::kStages; ++s) {
            mbar_init(smem_u32(&bars.kv_full[s]), 1);
            mbar_init(smem_u32(&bars.kv_empty[s]), 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(smem_u32(&bars.s_full[t]), 1);
            mbar_init(smem_u32(&bars.p_full[t]), 4);  // one arrival per softmax warp
            mbar_init(smem_u32(&bars.o_done[t]), 1);
        }
        mbar_init(smem_u32(&bars.v_need), 1);
        mbar_init(smem_u32(&bars.v_fixed), 1);
        mbar_init(smem_u32(&bars.drain), 1);
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        prefetch_map(&p.tm_q);
        prefetch_map(&p.tm_kpool);
        prefetch_map(&p.tm_vpool);
    }
    if (c.tile_rows < 128) {  // rows past the packed ones are never copied: finite values, so that their softmax stays quiet
        const int n = (128 - c.tile_rows) * 8;
        for (int i = threadIdx.x; i < 2 * Sh::kParts * n; i += kThreadsTc)
            *reinterpret_cast<uint4*>(c.smem + (i / n) * 16384 + c.tile_rows * 128 + (i % n) * 16) = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&bars.tmem_base))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    c.tmem = bars.tmem_base;
    if (p.n_splits == 1) pdl_trigger();
    pdl_wait();
    // tensor-memory columns: S_t at t*128, O_t at 256 + t*128; P_t aliases S_t (64 columns of bf16 pairs)

    c.seq_len = max(p.seq_lens[c.b], 0);
    c.M = p.q_lens ? p.q_lens[c.b] : p.M_max;
    c.M = min(max(c.M, 0), p.M_max);
    bool work = c.tok0 < c.M;                    // (uniform for the CTA)
    const bool one = kForm == kOneTile || (kForm == kBoth && c.M - c.tok0 <= c.tok_per_tile);  // one row tile

    // KV range of this split: an equal share of the sequence's 128-token tiles and the tile of the step's own tokens,
    // which comes last
    const int total_tiles = (c.seq_len + kTileTokens - 1) / kTileTokens;
    const uint32_t positions = (uint32_t)total_tiles + 1;  // at most 2^24 + 1, and at most 64 splits
    c.tile_begin = (int)(positions * (uint32_t)c.split / (uint32_t)p.n_splits);
    c.n_tiles = (int)(positions * (uint32_t)(c.split + 1) / (uint32_t)p.n_splits) - c.tile_begin;
    const bool last_split = c.split == p.n_splits - 1;
    c.n_ctx_tiles = c.n_tiles - (last_split ? 1 : 0);
    const int tile_end = c.tile_begin + c.n_ctx_tiles;
    // first tile whose V rows need zeroing past the valid tokens: a ragged last context tile, else the
    // tile of the step's own tokens (fewer than 128), else none
    const bool ragged_ctx = c.n_ctx_tiles > 0 && tile_end == total_tiles && (c.seq_len % kTileTokens) != 0;
    c.first_fix = ragged_ctx ? c.n_ctx_tiles - 1 : ((last_split && c.M < kTileTokens) ? c.n_ctx_tiles : c.n_tiles);

    if (work && c.n_tiles == 0) {
        // an empty split: publish (m = -inf, l = 0) so that the merge ignores it
        for (int r = threadIdx.x; r < p.rg_tiles * 128; r += kThreadsTc) {
            const size_t prow = (((size_t)c.lb * p.Hkv + c.h) * p.n_splits + c.split) * p.R_pad + c.rg * p.rg_tiles * 128 + r;
            p.part_ml[prow * 2] = -INFINITY;
            p.part_ml[prow * 2 + 1] = 0.f;
        }
        work = false;
    }

    if (work) {
        // Register budget: the control warpgroup (warps 0-3) gives registers to the two softmax warpgroups: 128 x 56 +
        // 256 x 224 = the 384 x 168 of the launch.
        if (warp == 0) {
            asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
            copy_q<D>(p, c, bars, one, lane);
            produce<D>(p, c, bars, one, lane);
        } else if (warp == 1) {
            asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
            one ? issue<D, true, kSplit>(p, c, bars, lane) : issue<D, false, kSplit>(p, c, bars, lane);
        } else if (warp == 2) {
            asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
            one ? fix_v<D, true>(p, c, bars, lane) : fix_v<D, false>(p, c, bars, lane);
        } else if (warp == 3) {
            asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        } else {
            asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
            one ? softmax<D, true, kSplit>(p, c, bars, warp, lane) : softmax<D, false, kSplit>(p, c, bars, warp, lane);
        }
    }

    // ---- teardown ----------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (p.n_splits > 1) pdl_trigger();
    if (warp == 1) {
        // after a give-up no new copy was issued; the few in flight (at most a ring of them) land within microseconds
        if (*(volatile int*)&bars.abort_flag) __nanosleep(1000000);
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(c.tmem) : "memory");
    }
}

// Log-sum-exp merge of the KV splits: D/4 threads per row, each owning four channels.  Bound by latency: the partial rows
// come from L2, so kMergeAhead of them are in flight per thread, requested before the splits' maxima are known, and a
// row's threads fetch the maxima and sums of as many splits side by side (one layer, 60 rows x 4 heads, 9 splits: 3.8 ->
// 2.3 us against four loads in flight behind a serial pass over the maxima).  Splits are added in order.
constexpr int kMergeThreads = 512;
constexpr int kMergeAhead = 8;
template <int D>
__global__ void __launch_bounds__(kMergeThreads) merge_tc_kernel(const __grid_constant__ TcParams p) {
    pdl_begin(p.pdl);
    constexpr int kRowThreads = D / 4;
    const int row_in_head = blockIdx.x * (kMergeThreads / kRowThreads) + threadIdx.x / kRowThreads;  // step token * G + query head
    const int h = blockIdx.y, lb = blockIdx.z, lane = threadIdx.x % kRowThreads;
    const int b = lb % p.batch;
    int M = p.q_lens ? p.q_lens[b] : p.M_max;
    M = min(max(M, 0), p.M_max);
    if (row_in_head >= M * p.G) return;
    const unsigned members = kRowThreads == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);  // the row's lanes
    const int j = row_in_head / p.G, g = row_in_head % p.G;
    const int tok_per_tile = 128 / p.G;
    const int r = j / tok_per_tile * 128 + j % tok_per_tile * p.G + g;  // its place in the packed row tiles
    const size_t row0 = ((size_t)lb * p.Hkv + h) * p.n_splits * p.R_pad + r;
    const float4* po = reinterpret_cast<const float4*>(p.part_o + row0 * D) + lane;
    const float2* ml = reinterpret_cast<const float2*>(p.part_ml) + row0;
    const size_t po_stride = (size_t)p.R_pad * kRowThreads;
    float4 buf[kMergeAhead];
#pragma unroll
    for (int u = 0; u < kMergeAhead; ++u)
        if (u < p.n_splits) buf[u] = po[u * po_stride];
    float m_all = -INFINITY;
    for (int s = lane; s < p.n_splits; s += kRowThreads) m_all = fmaxf(m_all, ml[(size_t)s * p.R_pad].x);
#pragma unroll
    for (int o = kRowThreads / 2; o > 0; o >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(members, m_all, o));
    float l_all = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < p.n_splits; c0 += kRowThreads) {  // a lane per split of this chunk
        float w_mine = 0.f, l_mine = 0.f;
        if (c0 + lane < p.n_splits) {
            const float2 v = ml[(size_t)(c0 + lane) * p.R_pad];
            if (v.x != -INFINITY) {  // an empty split's partial O was never written: weight 0, not used
                w_mine = ex2(v.x - m_all);
                l_mine = v.y * w_mine;
            }
        }
        for (int s0 = c0; s0 < min(c0 + kRowThreads, p.n_splits); s0 += kMergeAhead) {
#pragma unroll
            for (int u = 0; u < kMergeAhead; ++u) {
                const float w = __shfl_sync(members, w_mine, s0 - c0 + u, kRowThreads);
                l_all += __shfl_sync(members, l_mine, s0 - c0 + u, kRowThreads);
                if (s0 + u >= p.n_splits) break;
                if (w != 0.f) {
                    o.x = fmaf(buf[u].x, w, o.x);
                    o.y = fmaf(buf[u].y, w, o.y);
                    o.z = fmaf(buf[u].z, w, o.z);
                    o.w = fmaf(buf[u].w, w, o.w);
                }
            }
#pragma unroll
            for (int u = 0; u < kMergeAhead; ++u)
                if (s0 + kMergeAhead + u < p.n_splits) buf[u] = po[(size_t)(s0 + kMergeAhead + u) * po_stride];
        }
    }
    const size_t row = ((size_t)lb * p.M_max + j) * p.Hq + h * p.G + g;
    const float inv = 1.f / l_all;
    o.x *= inv; o.y *= inv; o.z *= inv; o.w *= inv;
    if (p.out_f32) {
        reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + row * D)[lane] = o;
    } else {
        uint2 w2;
        w2.x = pack_bf16(o.x, o.y);
        w2.y = pack_bf16(o.z, o.w);
        reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + row * D)[lane] = w2;
    }
    if (p.lse && lane == 0) p.lse[row] = fmaf(m_all, kLn2, logf(l_all));
}

template <int D, int kForm, bool kSplit>
specpv_status launch_form(const TcParams& p, int n_lb, cudaStream_t stream) {
    using Sh = Shape<D>;
    if (!set_smem_limit_once(reinterpret_cast<const void*>(attn_tc_kernel<D, kForm, kSplit>), Sh::kSmemBytes)) return SPECPV_ERR_CUDA;
    if (launch_pdl(attn_tc_kernel<D, kForm, kSplit>, p.n_splits * p.n_row_groups * p.Hkv * n_lb, kThreadsTc, Sh::kSmemBytes, stream, p) !=
        cudaSuccess)
        return SPECPV_ERR_CUDA;
    count_launch();
    return SPECPV_OK;
}

template <int D, bool kSplit>
specpv_status launch_kernels(const TcParams& p, int n_lb, cudaStream_t stream) {
    // per-sequence row counts, or a last row group of one tile, can bring both forms into one launch
    const bool both = p.rg_tiles == 2 && (p.q_lens || p.n_full_groups < p.n_row_groups);
    const specpv_status st = p.rg_tiles == 1 ? launch_form<D, kOneTile, kSplit>(p, n_lb, stream)
                             : both          ? launch_form<D, kBoth, kSplit>(p, n_lb, stream)
                                             : launch_form<D, kTwoTiles, kSplit>(p, n_lb, stream);
    if (st != SPECPV_OK) return st;
    if (p.n_splits > 1) {
        constexpr int rows = kMergeThreads / (D / 4);
        const dim3 grid((p.M_max * p.G + rows - 1) / rows, p.Hkv, n_lb);
        if (launch_pdl_if(merge_tc_kernel<D>, grid, kMergeThreads, 0, stream, p) != cudaSuccess)
            return SPECPV_ERR_CUDA;
        count_launch();
    }
    return SPECPV_OK;
}

// Time until `n_short` CTAs of `t_short` each, started behind `n_long` of `t_long`, are done on 148 SMs of one CTA each.
double cta_makespan(long long n_long, double t_long, long long n_short, double t_short) {
    constexpr long long kSms = 148;
    const long long q = n_long / kSms, more = n_long % kSms;  // `more` SMs take one long CTA more than the others
    const double early = q * t_long, late = early + (more ? t_long : 0.0);
    if (n_short == 0) return late;
    double end = 1e300;
    for (int on_early = 0; on_early < 2; ++on_early)  // the last short CTA ends on one kind of SM or the other
        for (long long k = 1; k <= n_short / kSms + (long long)(t_long / t_short) + 2; ++k) {
            const double t = (on_early ? early : late) + k * t_short;
            const long long done = more * (t >= late ? (long long)((t - late) / t_short + 1e-9) : 0) +
                                   (kSms - more) * (t >= early ? (long long)((t - early) / t_short + 1e-9) : 0);
            if (done < n_short) continue;
            const double all = t > late ? t : late;
            end = all < end ? all : end;
            break;
        }
    return end;
}

}  // namespace

bool attention_tc_supported(const AttnArgs& a) {
    if (a.g.dtype != SPECPV_DTYPE_BF16 || (a.g.d != 128 && a.g.d != 64) || (a.g.bs != 64 && a.g.bs != 32 && a.g.bs != 16)) return false;
    if (a.g.G > 128) return false;
    if (a.M_max > kMaxQTokens) return false;
    // row coordinates of the pool tensor map must fit in a positive int32
    const unsigned long long rows = (unsigned long long)a.g.n_layers * a.n_pages * a.g.Hkv * (unsigned long long)a.g.bs;
    if (rows >= 0x7FFFFF00ull) return false;
    return get_encode_fn() != nullptr;
}

specpv_status launch_attention_tc(const AttnArgs& a, cudaStream_t stream) {
    TcParams p{};
    const int G = a.g.G, Hq = a.g.Hq, Hkv = a.g.Hkv;
    const uint64_t d = (uint64_t)a.g.d;
    const uint64_t step_tokens = (uint64_t)a.n_layers * a.batch * a.M_max;
    const bool pair = attention_pair_wanted(a);
    if (pair) {
        uint64_t dims[3] = {d, (uint64_t)Hq, step_tokens};
        uint64_t strides[2] = {2 * d, (uint64_t)Hq * 2 * d};
        uint32_t box[3] = {64, (uint32_t)G, (uint32_t)(128 / G)};
        if (!encode_map(&p.tm_q, a.q, 3, dims, strides, box)) return SPECPV_ERR_CUDA;
    } else {
        // Four dimensions, so that rows past a sequence's M_max tokens arrive as zeros: they cost the tensor pipe less power than
        // the next layer's queries (64K tokens x 36 layers: 38 rows per head 2078 -> 2012 us, 48 rows 2127 -> 2074, 13 rows 1399 -> 1357).
        uint64_t dims[4] = {d, (uint64_t)Hq, (uint64_t)a.M_max, (uint64_t)a.n_layers * a.batch};
        uint64_t strides[3] = {2 * d, (uint64_t)Hq * 2 * d, (uint64_t)a.M_max * Hq * 2 * d};
        uint32_t box[4] = {64, (uint32_t)G, (uint32_t)(128 / G), 1};
        if (!encode_map(&p.tm_q, a.q, 4, dims, strides, box)) return SPECPV_ERR_CUDA;
    }
    {
        uint64_t dims[3] = {d, (uint64_t)Hkv, step_tokens};
        uint64_t strides[2] = {2 * d, (uint64_t)Hkv * 2 * d};
        uint32_t box[3] = {64, 1, pair ? 64u : 8u};
        if (!encode_map(&p.tm_knew, a.k_new, 3, dims, strides, box)) return SPECPV_ERR_CUDA;
        if (!encode_map(&p.tm_vnew, a.v_new, 3, dims, strides, box)) return SPECPV_ERR_CUDA;
    }
    const uint64_t pool_rows = (uint64_t)a.g.n_layers * a.n_pages * Hkv * (uint64_t)a.g.bs;
    if (pair) {
        uint64_t dims[2] = {d, pool_rows};
        uint64_t strides[1] = {2 * d};
        uint32_t box[2] = {64, (uint32_t)a.g.bs};
        if (!encode_map(&p.tm_kpool, a.k_pool, 2, dims, strides, box)) return SPECPV_ERR_CUDA;
        if (!encode_map(&p.tm_vpool, a.v_pool, 2, dims, strides, box)) return SPECPV_ERR_CUDA;
    } else {  // (64 channels, 8 tokens, parts, groups of 8 tokens): a page's box lands group by group, its parts side by side
        uint64_t dims[4] = {64, 8, d / 64, pool_rows / 8};
        uint64_t strides[3] = {2 * d, 128, 16 * d};
        uint32_t box[4] = {64, 8, (uint32_t)d / 64, (uint32_t)a.g.bs / 8};
        if (!encode_map(&p.tm_kpool, a.k_pool, 4, dims, strides, box)) return SPECPV_ERR_CUDA;
        if (!encode_map(&p.tm_vpool, a.v_pool, 4, dims, strides, box)) return SPECPV_ERR_CUDA;
    }
    p.tree_mask = a.tree_mask; p.q_lens = a.q_lens; p.block_table = a.block_table; p.seq_lens = a.seq_lens;
    p.out = a.out; p.lse = a.lse; p.workspace = a.workspace;
    p.layer0 = a.layer0; p.batch = a.batch; p.M_max = a.M_max; p.mask_words = a.mask_words;
    p.Hq = Hq; p.Hkv = Hkv; p.G = G; p.max_blocks = a.max_blocks; p.n_pages = a.n_pages;
    p.out_f32 = a.g.out_f32;
    p.bs = a.g.bs;
    p.pool_rows = (uint32_t)pool_rows;
    p.scale_log2 = a.g.scale * kLog2e;
    // kSplit: what the float32 factor leaves out, and the mean of what the tensor core cuts off a dot product of d channels, which it
    // sums 16 at a time and truncates each time (measured, of the sum: 4.6e-8 to 8.3e-8 at 64 channels, 8.9e-8 to 13.8e-8 at
    // 128, the more the more alike the terms are).  Without this term every log-sum-exp comes out 5e-8 to 6e-8 of itself too
    // small: rms error 6.1e-8 and 7.3e-8 at 64 and 128 channels, 3.3e-8 and 3.5e-8 with it.  The term is positive, as the products
    // of masked scores, -infinity, need it to be: scale_log2 is at most 2^-24 = 6.0e-8 of itself, less the 1.3e-8 that
    // kLog2e is too small by, above the exact factor, and 6.4e-8 are added (and where all of this underflows, the smallest float).
    p.scale_log2_lo = (float)((double)a.g.scale * 1.4426950408889634 * (1.0 + 1.0e-9 * a.g.d) - (double)p.scale_log2);
    if (!(p.scale_log2_lo > 0.f)) p.scale_log2_lo = 1.4e-45f;

    if (pair) {
        p.n_row_groups = (a.M_max * G + 255) / 256;
        p.R_pad = p.n_row_groups * 256;
        return launch_attention_pair(p, a, stream);
    }
    // Row tiles per CTA and KV splits, by a cost model in microseconds (one CTA per SM).  A tile costs 0.9 with one row tile
    // per CTA (alternate streams) and 1.5 with two (the same contractions for half the K/V traffic).  A CTA pays 7 for
    // set-up, first tile and drain; splitting adds the partial results (1.5 / 4 per CTA, and their bytes) and the merge launch.
    // Two row tiles are the better form when there are CTAs enough; one row tile gives twice the CTAs where a launch
    // cannot fill the SMs otherwise (one layer, 8 KV heads, 60 rows x 4: 4096 tokens 20.0 -> 18.6 us, 16384 tokens
    // 32.5 -> 29.2 us).  Down to one tile per CTA pays (24 rows x 4, 2048 tokens: 15.8 / 15.1 / 14.2 us at 6 / 9 / 18
    // splits).  A last row group of one tile makes shorter CTAs, which come last in the grid (64K tokens x 36 layers,
    // 90 rows x 4: 4100 -> 3690 us).
    const int tok_per_tile = 128 / G, row_tiles = (a.M_max + tok_per_tile - 1) / tok_per_tile;
    const int n_units = Hkv * a.n_layers * a.batch;
    const int positions = (a.max_seq_len + kTileTokens - 1) / kTileTokens + 1;  // context tiles + the tile of the step's own tokens
    const double row_bytes = (double)n_units * a.M_max * G * (a.g.d + 2) * sizeof(float);  // partial results of a split
    const double tile_bytes = (double)n_units * 128 * (a.g.d + 2) * sizeof(float);
    // The partial rows are stored 32 bytes at a time and a workspace need only be 16-byte aligned: they start at the next multiple of
    // 32, and the 16 bytes before it are not counted as scratch.
    char* ws = reinterpret_cast<char*>(a.workspace) + a.partial_off;
    const size_t skip = (32 - (reinterpret_cast<uintptr_t>(ws) & 31)) & 31;
    const double scratch = (double)a.partial_bytes - (double)skip;
    double best_cost = 1e30;
    for (int rg_tiles = row_tiles > 1 ? 2 : 1; rg_tiles >= 1; --rg_tiles) {
        const int groups = (row_tiles + rg_tiles - 1) / rg_tiles, full = row_tiles / rg_tiles;
        for (int s = 1; s <= 64 && s <= positions; ++s) {
            if (s > 1 && tile_bytes * s * groups * rg_tiles > scratch) break;
            const int tiles = (positions + s - 1) / s;
            const double t1 = 7.0 + 0.9 * tiles + (s > 1 ? 1.5 : 0.0), t2 = 7.0 + 1.5 * tiles + (s > 1 ? 4.0 : 0.0);
            const long long n_long = (long long)n_units * s * full, n_short = (long long)n_units * s * (groups - full);
            double cost = cta_makespan(n_long, rg_tiles == 2 ? t2 : t1, n_short, t1);
            if (s > 1) cost += 3.0 + row_bytes * s * 2.0 / 5.3e6;  // written and read through L2 at 5.3 TB/s
            if (cost < best_cost) {
                best_cost = cost;
                p.n_splits = s;
                p.rg_tiles = rg_tiles;
            }
        }
    }
    p.n_row_groups = (row_tiles + p.rg_tiles - 1) / p.rg_tiles;
    p.n_full_groups = row_tiles / p.rg_tiles;
    p.n_full_units = n_units * p.n_full_groups;
    p.R_pad = p.n_row_groups * p.rg_tiles * 128;
    p.part_o = reinterpret_cast<float*>(ws + skip);
    p.part_ml = reinterpret_cast<float*>(ws + skip + (size_t)n_units * p.n_splits * p.R_pad * a.g.d * sizeof(float));

    const int n_lb = a.n_layers * a.batch;
    if (a.g.d == 64) return launch_kernels<64, true>(p, n_lb, stream);
    return 128 % G == 0 ? launch_kernels<128, false>(p, n_lb, stream) : launch_kernels<128, true>(p, n_lb, stream);
}

}  // namespace specpv
