// Cache-management kernels of the SpecPV verification path (paper Section 3.2-3.3):
// block key summaries (Eq. 1), block scores (Eq. 2-3), the retained-block selection, the gather
// that rebuilds the partial cache, and the commit of accepted tokens.
#include <math.h>

#include "common.cuh"
#include "aux_kernels.cuh"
#include "tc_common.cuh"

namespace specpv {

namespace {

// ---------------------------------------------------------------------------------------------
// Eq. 1: Kmax/Kmin per block.  A warp owns one (block, KV head): a lane keeps one 16-byte chunk of channels and every
// (32 / chunks)-th token, kSumLoads loads in flight, max and min taken on packed pairs (both exact, so neither the
// packing nor the order matters), the token lanes combined by shuffles.  No shared memory and no barrier: the kernel is
// a pure stream, bound by HBM.  6.4 GB of keys (96K tokens x 32 layers x 8 heads): 941 us = 6.8 TB/s against 1872 us for
// a CTA per (block, head) that widened to float32 and reduced through shared memory; a copy runs at 6.5 TB/s.
// grid = (blocks touched, head groups, layers x seqs).
// ---------------------------------------------------------------------------------------------
constexpr int kSumWarps = 8;   // KV heads per CTA: the heads of a page are contiguous
constexpr int kSumLoads = 16;  // 16-byte loads in flight per lane

// NaN operands lose against numbers, like fmaxf / fminf.
__device__ __forceinline__ uint32_t packed_max(uint32_t a, uint32_t b, __nv_bfloat16) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t packed_min(uint32_t a, uint32_t b, __nv_bfloat16) {
    uint32_t r;
    asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ uint32_t packed_max(uint32_t a, uint32_t b, float) {
    return __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b)));
}
__device__ __forceinline__ uint32_t packed_min(uint32_t a, uint32_t b, float) {
    return __float_as_uint(fminf(__uint_as_float(a), __uint_as_float(b)));
}

// A lane's running maximum and minimum of one 16-byte chunk of channels.
template <typename T>
struct SummaryAcc {
    static constexpr uint32_t kNegInf = sizeof(T) == 2 ? 0xFF80FF80u : 0xFF800000u;
    static constexpr uint32_t kPosInf = kNegInf & (sizeof(T) == 2 ? 0x7FFF7FFFu : 0x7FFFFFFFu);
    uint32_t mx[4] = {kNegInf, kNegInf, kNegInf, kNegInf}, mn[4] = {kPosInf, kPosInf, kPosInf, kPosInf};
    __device__ __forceinline__ void take(const uint4& v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            mx[e] = packed_max(mx[e], w[e], T());
            mn[e] = packed_min(mn[e], w[e], T());
        }
    }
    __device__ __forceinline__ void combine(int chunks) {  // over the lanes that hold the same chunk
        for (int o = 16; o >= chunks; o >>= 1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                mx[e] = packed_max(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o), T());
                mn[e] = packed_min(mn[e], __shfl_xor_sync(0xffffffffu, mn[e], o), T());
            }
        }
    }
    __device__ __forceinline__ void store(void* kmax, void* kmin, int aligned, size_t o) const {  // o: in 16-byte chunks
        const uint4 vx = make_uint4(mx[0], mx[1], mx[2], mx[3]), vn = make_uint4(mn[0], mn[1], mn[2], mn[3]);
        if (aligned) {
            reinterpret_cast<uint4*>(kmax)[o] = vx;
            reinterpret_cast<uint4*>(kmin)[o] = vn;
        } else {
            constexpr int kChunk = 16 / (int)sizeof(T);
#pragma unroll
            for (int e = 0; e < kChunk; ++e) {
                reinterpret_cast<T*>(kmax)[o * kChunk + e] = reinterpret_cast<const T*>(&vx)[e];
                reinterpret_cast<T*>(kmin)[o * kChunk + e] = reinterpret_cast<const T*>(&vn)[e];
            }
        }
    }
};

template <typename T>
__global__ void __launch_bounds__(32 * kSumWarps) summaries_kernel(SummaryParams p) {
    pdl_begin(p.pdl);
    const int lane = threadIdx.x & 31;
    const int h = blockIdx.y * kSumWarps + (threadIdx.x >> 5), lb = blockIdx.z;
    const int b = lb % p.batch, l = lb / p.batch;
    const int seq_len = p.seq_lens[b];
    const int begin = p.tok_begin ? p.tok_begin[b] : 0;
    const int i = max(begin, 0) / p.bs + blockIdx.x;
    if (h >= p.Hkv || (size_t)i * p.bs >= (size_t)seq_len || i >= p.max_blocks) return;
    const int n_valid = min(p.bs, seq_len - i * p.bs);
    const int page = p.block_table[(size_t)b * p.max_blocks + i];
    if (page < 0 || page >= p.n_pages) {
        if (lane == 0) record_fault(p.workspace, SPECPV_ERR_BAD_BLOCK_TABLE, b, i, page, l);
        return;
    }
    const int chunks = p.d * (int)sizeof(T) / 16;  // 16-byte chunks per token row: 8, 16 or 32
    const int tok_lanes = 32 / chunks;             // tokens read side by side
    const int chunk = lane % chunks, tl = lane / chunks;
    const uint4* k = reinterpret_cast<const uint4*>(reinterpret_cast<const T*>(p.k_pool) +
                                                    (((size_t)(p.layer0 + l) * p.n_pages + page) * p.Hkv + h) * p.bs * p.d) + chunk;
    SummaryAcc<T> acc;
    for (int t0 = 0; t0 < n_valid; t0 += kSumLoads * tok_lanes) {
        uint4 buf[kSumLoads];
#pragma unroll
        for (int u = 0; u < kSumLoads; ++u)  // past the last valid token: that token again, which changes nothing
            buf[u] = k[(size_t)min(t0 + u * tok_lanes + tl, n_valid - 1) * chunks];
#pragma unroll
        for (int u = 0; u < kSumLoads; ++u) acc.take(buf[u]);
    }
    acc.combine(chunks);
    if (tl == 0)
        acc.store(p.kmax, p.kmin, p.aligned, ((((size_t)(p.layer0 + l) * p.batch + b) * p.Hkv + h) * p.max_blocks + i) * chunks + chunk);
}

// ---------------------------------------------------------------------------------------------
// Eq. 2-3 (SIMT form): a warp owns kBlocks blocks, whose summaries are staged in shared memory as float32 and read as broadcasts, a
// lane the query rows lane, lane + 32, .. of the group, staged kScoreRows at a time; a block's results are added over the lanes by
// shuffles.  Up to kScoreFewRows rows, eight lanes share a row (kParts) and take every eighth four channels.  Bound by latency on
// the small shapes it serves: one block per warp spreads 75 blocks of two heads over 20 CTAs (a lane per block and 32 blocks per CTA left
// them on 6: 128 rows of 64 channels 18.6 -> 6.6 us, 33 blocks and 64 rows 10.3 -> 4.1); four blocks per warp read the rows once for
// four where the launch has CTAs enough.  Larger ones, us, a lane per block / four blocks per warp with a lane per row, summaries loaded
// 2 or 4 bytes at a time / this form: 240 rows of 128, 512 blocks x 32 lists 110 / 104 / 102; 64 rows of 128, 512 x 256 233 / 204 / 179; 4 rows
// of 128, 2048 x 128 203 / 217 / 94, 512 x 32 12.6 / 18.1 / 8.8; 5 rows of 128 (bfloat16), 1024 x 64 45 / 56 / 34; 2 rows of 64 (bfloat16),
// 1000 x 64 17.7 / 25.4 / 16.2.  grid = (block groups, Hkv, layers x seqs).
// ---------------------------------------------------------------------------------------------
constexpr int kScoreWarps = 8;
constexpr int kScoreRows = 64;     // query rows staged at a time
constexpr int kScoreFewRows = 16;  // .. where eight lanes share a row

// 16 bytes of storage elements as float32
__device__ __forceinline__ void store_floats(float* dst, uint4 v, float) { *reinterpret_cast<uint4*>(dst) = v; }
__device__ __forceinline__ void store_floats(float* dst, uint4 v, __nv_bfloat16) {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(v.x << 16, v.x & 0xffff0000u, v.y << 16, v.y & 0xffff0000u);
    reinterpret_cast<uint4*>(dst)[1] = make_uint4(v.z << 16, v.z & 0xffff0000u, v.w << 16, v.w & 0xffff0000u);
}

// Registers: eight lanes to a row need no unrolling but room for the loads (four blocks: 80; 94 -> 217 us at 64, 114 with two steps unrolled);
// four blocks of 128 channels get what three CTAs leave each other (64 rows, 512 blocks x 256 lists 205 -> 179 us).
template <typename T, int D, int kBlocks, int kParts>
__global__ void __launch_bounds__(32 * kScoreWarps, kParts > 1 ? 1 : kBlocks == 4 && D == 128 ? 3 : 0) scores_simt_kernel(ScoreParams p) {
    pdl_begin(p.pdl);
    constexpr int kPitch = D + 4, kCtaBlocks = kScoreWarps * kBlocks;  // pitch: a warp's 16-byte reads of 32 rows meet no bank twice
    extern __shared__ __align__(16) float smem[];
    constexpr int kRows = kParts == 1 ? kScoreRows : kScoreFewRows;
    float* rows_s = smem;                          // [kRows][kPitch]
    float* sums_s = rows_s + kRows * kPitch;       // [blocks][2][D]: Kmax, Kmin
    const int h = blockIdx.y, lb = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = lb % p.batch, l = lb / p.batch;
    const int seq_len = p.seq_lens[b];
    const int nb = (seq_len + p.bs - 1) / p.bs;
    const int blk0 = blockIdx.x * kCtaBlocks;
    if (blk0 >= nb) return;
    int M = p.q_lens ? p.q_lens[b] : p.M_max;
    M = min(max(M, 0), p.M_max);
    int row_begin = 0, row_end = M * p.G;  // rows r = j * G + g
    if (p.reduce == SPECPV_REDUCE_LAST) {
        int last = p.last_query ? p.last_query[b] : 0;
        last = min(max(last, 0), max(M - 1, 0));
        row_begin = last * p.G;
        row_end = row_begin + p.G;
    }
    const size_t sum_base = ((((size_t)(p.layer0 + l) * p.batch + b) * p.Hkv + h) * p.max_blocks) * D;
    const T* kmax = reinterpret_cast<const T*>(p.kmax) + sum_base;
    const T* kmin = reinterpret_cast<const T*>(p.kmin) + sum_base;
    if (((reinterpret_cast<uintptr_t>(kmax) | reinterpret_cast<uintptr_t>(kmin)) & 15) == 0) {  // (uniform; summaries may start anywhere)
        constexpr int kVec = 16 / (int)sizeof(T);
#pragma unroll
        for (int e = tid; e < kCtaBlocks * D / kVec; e += 32 * kScoreWarps) {
            const int bi = e / (D / kVec), c = e % (D / kVec) * kVec, i = blk0 + bi;
            uint4 hi = make_uint4(0, 0, 0, 0), lo = hi;
            if (i < nb) {
                hi = *reinterpret_cast<const uint4*>(kmax + (size_t)i * D + c);
                lo = *reinterpret_cast<const uint4*>(kmin + (size_t)i * D + c);
            }
            store_floats(sums_s + (bi * 2) * D + c, hi, T());
            store_floats(sums_s + (bi * 2 + 1) * D + c, lo, T());
        }
    } else {
#pragma unroll 4
        for (int e = tid; e < kCtaBlocks * D; e += 32 * kScoreWarps) {
            const int bi = e / D, c = e % D, i = blk0 + bi;
            sums_s[(bi * 2) * D + c] = i < nb ? to_float(kmax[(size_t)i * D + c]) : 0.f;
            sums_s[(bi * 2 + 1) * D + c] = i < nb ? to_float(kmin[(size_t)i * D + c]) : 0.f;
        }
    }
    const T* q = reinterpret_cast<const T*>(p.q) + (size_t)lb * p.M_max * p.Hq * D;
    const bool reduce_max = p.reduce == SPECPV_REDUCE_MAX;
    float red[kBlocks];
#pragma unroll
    for (int k = 0; k < kBlocks; ++k) red[k] = reduce_max ? -INFINITY : 0.f;
    for (int r0 = row_begin; r0 < row_end; r0 += kRows) {
        if (r0 != row_begin) __syncthreads();  // the rows before these have been read
        const int n_rows = min(kRows, row_end - r0);
#pragma unroll 4
        for (int r = warp; r < n_rows; r += kScoreWarps) {
            const T* src = q + ((size_t)((r0 + r) / p.G) * p.Hq + h * p.G + (r0 + r) % p.G) * D;
#pragma unroll
            for (int c = lane; c < D; c += 32) rows_s[r * kPitch + c] = to_float(src[c]);
        }
        __syncthreads();
        for (int r = lane / kParts; kParts == 1 ? r < n_rows : r - lane / kParts < n_rows; r += 32 / kParts) {
            const int c0 = kParts == 1 ? 0 : 4 * (lane % kParts);  // the lane's first channels
            const float* row = rows_s + (kParts == 1 ? r : min(r, n_rows - 1)) * kPitch;
            const float* sums = sums_s + warp * kBlocks * 2 * D;
            float dmax[kBlocks], dmin[kBlocks];
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) dmax[k] = dmin[k] = 0.f;
            if (p.score_mode == 0) {
#pragma unroll (kParts == 1 ? 4 : 1)
                for (int c = c0; c < D; c += 4 * kParts) {
                    const float4 qv = *reinterpret_cast<const float4*>(row + c);
#pragma unroll
                    for (int k = 0; k < kBlocks; ++k) {
                        const float4 a = *reinterpret_cast<const float4*>(sums + k * 2 * D + c);
                        const float4 bb = *reinterpret_cast<const float4*>(sums + (k * 2 + 1) * D + c);
                        dmax[k] = fmaf(qv.w, a.w, fmaf(qv.z, a.z, fmaf(qv.y, a.y, fmaf(qv.x, a.x, dmax[k]))));
                        dmin[k] = fmaf(qv.w, bb.w, fmaf(qv.z, bb.z, fmaf(qv.y, bb.y, fmaf(qv.x, bb.x, dmin[k]))));
                    }
                }
            } else {
                // channel-wise form: a channel with q_c >= 0 takes Kmax_c, one with q_c < 0 takes Kmin_c
                // (Kmax_c >= Kmin_c), so the score is one dot product with a per-channel choice of operand
#pragma unroll (kParts == 1 ? 4 : 1)
                for (int c = c0; c < D; c += 4 * kParts) {
                    const float4 qv = *reinterpret_cast<const float4*>(row + c);
#pragma unroll
                    for (int k = 0; k < kBlocks; ++k) {
                        const float4 a = *reinterpret_cast<const float4*>(sums + k * 2 * D + c);
                        const float4 bb = *reinterpret_cast<const float4*>(sums + (k * 2 + 1) * D + c);
                        dmax[k] = fmaf(qv.x, qv.x < 0.f ? bb.x : a.x, dmax[k]);
                        dmax[k] = fmaf(qv.y, qv.y < 0.f ? bb.y : a.y, dmax[k]);
                        dmax[k] = fmaf(qv.z, qv.z < 0.f ? bb.z : a.z, dmax[k]);
                        dmax[k] = fmaf(qv.w, qv.w < 0.f ? bb.w : a.w, dmax[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < kBlocks; ++k) dmin[k] = dmax[k];
            }
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) {
#pragma unroll
                for (int o = kParts / 2; o > 0; o >>= 1) {
                    dmax[k] += __shfl_xor_sync(0xffffffffu, dmax[k], o);
                    dmin[k] += __shfl_xor_sync(0xffffffffu, dmin[k], o);
                }
                if (kParts > 1 && (r >= n_rows || c0 != 0)) continue;
                const float s = fmaxf(dmax[k], dmin[k]);
                red[k] = reduce_max ? fmaxf(red[k], s) : red[k] + s;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kBlocks; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float other = __shfl_xor_sync(0xffffffffu, red[k], o);
            red[k] = reduce_max ? fmaxf(red[k], other) : red[k] + other;
        }
        const int i = blk0 + warp * kBlocks + k;
        if (lane == 0 && i < nb)
            p.scores[((size_t)lb * p.Hkv + h) * p.max_blocks + i] = reduce_max ? red[k] : red[k] / (float)(row_end - row_begin);
    }
}

// ---------------------------------------------------------------------------------------------
// Selection: one CTA per (layer, sequence, KV head).  A candidate's score becomes a 32-bit key whose unsigned order is
// "score ascending, NaN first".  The key T of the k-th best candidate starts with the bits that all keys share (those of the smallest
// and the largest) and is found two bits at a time from there, by counting the keys (in registers) that reach each of three
// thresholds, until a threshold is met by k candidates exactly or all bits are known; after kSelectSteps steps the range of the keys
// that are still undecided is looked at again, which ends the search among equal scores.  Then an ordered compaction writes
// sink | kept candidates | local in ascending order, the candidates of key T that are still to be taken by lowest index.
// Bound by latency: a count and one barrier per step, and the fetch of its code, which follows other kernels: no more keys per
// thread, each of them code, than the lists need.  us per call, repeated calls, scores of one sign, against a histogram per digit of
// 11 bits / this search from the top bit, without a second look and with more code: 29 candidates x 2 lists 6.5 / 5.1 -> 3.3, 509 x 256
// 11.4 / 8.4 -> 6.0, 2045 x 256 13.2 / 12.9 -> 9.2 (with many ties 13.3 / 15.6 -> 7.7), 3837 x 128 11.5 / 13.9 -> 9.0, 4090 x 256
// 15.6 / 16.4 -> 13.9, 8189 x 256 31.8 / 38.3 -> 20.2, 16300 x 64 44.8 / 27.0 -> 22.5, 65000 x 32 223 / 140 -> 139.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t select_key(float score) {
    const uint32_t bits = __float_as_uint(score);
    if (score != score) return 0u;              // NaN ranks below every number
    if (score == 0.f) return 0x80000000u;       // -0 and +0 tie
    return (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
}

// Steps between two looks at the range of the undecided keys: most lists are decided after ten from the top bit.  (2045 x 256, one sign /
// many ties, measured with more code: 4 steps 11.2 / 9.5 us, 8 10.9 / 9.0, 16 10.4 / 13.2.)  Where keys are formed again for each step a look costs as much
// as a step: none at the start, and later than most lists need.
constexpr int kSelectSteps = 8, kSelectStepsTail = 12;

// kSelectKeys: a thread's keys stay in registers; those that the largest form has no room for are formed again from the scores.
// Registers: without a minimum of one CTA per SM the compiler stops at 32 and the loads wait for one another (2045 x 256: 9.2 -> 11.9 us);
// 16 keys in 512 threads leave room for two (8189 x 256: 26.3 -> 20.2).
template <int kSelectThreads, int kSelectKeys, bool kTail = false>
__global__ void __launch_bounds__(kSelectThreads, kSelectThreads == 512 && kSelectKeys == 16 ? 2 : 1) select_kernel(SelectParams p) {
    pdl_begin(p.pdl);
    constexpr int kWarps = kSelectThreads / 32, kCounts = kSelectKeys * kWarps;
    static_assert(32 * kSelectKeys < 1024 && kCounts % 32 == 0 && kCounts * 32 < 65536, "packed counts");
    __shared__ int4 s_reach[3];         // candidates that reach the thresholds of a step
    __shared__ uint2 s_range[kWarps];   // smallest and largest undecided key of each warp
    __shared__ unsigned s_counts[kCounts];  // per (round, warp): candidates above T | of key T << 16, then the sums of those before
    __shared__ unsigned s_total;        // ... and of all of them
    const int h = blockIdx.x, b = blockIdx.y, l = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t* idx = p.idx + (((size_t)l * p.batch + b) * p.Hkv + h) * p.budget_blocks;
    const int seq_len = p.seq_lens[b];
    const int nb = min((seq_len + p.bs - 1) / p.bs, p.max_blocks);
    const float* scores = p.scores + (((size_t)l * p.batch + b) * p.Hkv + h) * p.max_blocks;
    // share_heads: the score of a block is the float32 sum over the KV heads in head order, scaled by 1/Hkv (every CTA
    // of a layer computes the same sums and therefore the same list)
    const float* scores_h0 = p.scores + ((size_t)l * p.batch + b) * p.Hkv * p.max_blocks;
    const float inv_heads = 1.f / (float)p.Hkv;
    auto score_at = [&](int i) {
        if (!p.share_heads) return scores[i];
        float acc = 0.f;
        for (int hh = 0; hh < p.Hkv; ++hh) acc += scores_h0[(size_t)hh * p.max_blocks + i];
        return acc * inv_heads;
    };
    const int count = min(nb, p.budget_blocks);
    if (l == 0 && h == 0 && tid == 0) p.count[b] = count;
    if (nb <= p.budget_blocks) {
        for (int i = tid; i < nb; i += kSelectThreads) idx[i] = i;
        return;
    }
    const int lo = p.sink_blocks, hi = nb - p.local_blocks;
    const int k = p.budget_blocks - p.sink_blocks - p.local_blocks;

    // a thread's candidates: lo + tid, lo + tid + kSelectThreads, ...
    uint32_t keys[kSelectKeys];
    const int rounds = min((hi - lo + kSelectThreads - 1) / kSelectThreads, kSelectKeys);  // (no test of it where most keys are used)
    const int tail0 = lo + kSelectKeys * kSelectThreads;  // candidates from here on are not in registers
    uint32_t smallest = 0xffffffffu, largest = 0u;        // of this thread's undecided keys
    float own[kSelectKeys];  // their scores: as score_at, all loads of a head in flight together
    if (!p.share_heads) {
#pragma unroll
        for (int e = 0; e < kSelectKeys; ++e) {
            const int i = lo + tid + e * kSelectThreads;
            own[e] = i < hi ? scores[i] : 0.f;
        }
    } else {
#pragma unroll
        for (int e = 0; e < kSelectKeys; ++e) own[e] = 0.f;
#pragma unroll 2
        for (int hh = 0; hh < p.Hkv; ++hh)
#pragma unroll
            for (int e = 0; e < kSelectKeys; ++e) {
                const int i = lo + tid + e * kSelectThreads;
                own[e] += i < hi ? scores_h0[(size_t)hh * p.max_blocks + i] : 0.f;
            }
#pragma unroll
        for (int e = 0; e < kSelectKeys; ++e) own[e] *= inv_heads;
    }
#pragma unroll
    for (int e = 0; e < kSelectKeys; ++e) {
        const bool in = lo + tid + e * kSelectThreads < hi;
        keys[e] = in ? select_key(own[e]) : 0u;  // 0 reaches no threshold
        smallest = in ? min(smallest, keys[e]) : smallest;
        largest = max(largest, keys[e]);
    }
    const bool has_tail = kTail && tail0 < hi;
    if (has_tail) {
        smallest = 0u;
        largest = 0xffffffffu;
    }
    if (tid < 3) s_reach[tid] = make_int4(0, 0, 0, 0);
    uint32_t T;        // key of the k-th best candidate, the bits found so far
    int n_above = 0;   // candidates whose bits found so far are above T's
    int ties = -1;     // candidates of key T to take
    int at = 0;
#pragma unroll 1
    for (;;) {
        // the bits that all undecided keys share are T's
        smallest = __reduce_min_sync(0xffffffffu, smallest);
        largest = __reduce_max_sync(0xffffffffu, largest);
        if (lane == 0) s_range[warp] = make_uint2(smallest, largest);
        __syncthreads();
        const uint2 range = s_range[lane % kWarps];
        smallest = __reduce_min_sync(0xffffffffu, range.x);
        largest = __reduce_max_sync(0xffffffffu, range.y);
        T = smallest;
        if (smallest >= largest) break;  // one key is left
        int shift = (31 - __clz(smallest ^ largest)) & ~1;
        T &= ~((4u << shift) - 1u);
        const int stop = max(shift - 2 * (has_tail ? kSelectStepsTail : kSelectSteps), -2);
#pragma unroll 1
        for (; shift > stop; shift -= 2, at = at == 2 ? 0 : at + 1) {
            const uint32_t t1 = T + (1u << shift), t2 = T + (2u << shift), t3 = T + (3u << shift);
            unsigned c = 0;  // three counts of ten bits
#pragma unroll
            for (int e = 0; e < kSelectKeys; ++e)
                if (kSelectKeys > 8 || e < rounds) c += (keys[e] >= t1 ? 1u : 0u) + (keys[e] >= t2 ? 1u << 10 : 0u) + (keys[e] >= t3 ? 1u << 20 : 0u);
            c = __reduce_add_sync(0xffffffffu, c);
            int mine = lane < 3 ? (c >> (10 * lane)) & 1023u : 0;  // lane j: candidates of this warp that reach threshold j
            if (has_tail) {
                int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll 4
                for (int i = tail0 + tid; i < hi; i += kSelectThreads) {
                    const uint32_t key = select_key(score_at(i));
                    c1 += key >= t1;
                    c2 += key >= t2;
                    c3 += key >= t3;
                }
                c1 = __reduce_add_sync(0xffffffffu, c1);
                c2 = __reduce_add_sync(0xffffffffu, c2);
                c3 = __reduce_add_sync(0xffffffffu, c3);
                mine += lane == 0 ? c1 : lane == 1 ? c2 : c3;
            }
            if (lane < 3 && mine) atomicAdd(&s_reach[at].x + lane, mine);
            __syncthreads();
            const int4 reach = s_reach[at];
            if (tid == 0) s_reach[at == 0 ? 2 : at - 1] = make_int4(0, 0, 0, 0);  // read before this step's barrier, used behind the next one
            int reached;
            if (reach.z >= k) {
                T = t3;
                reached = reach.z;
            } else if (reach.y >= k) {
                T = t2;
                reached = reach.y;
                n_above = reach.z;
            } else if (reach.x >= k) {
                T = t1;
                reached = reach.x;
                n_above = reach.y;
            } else {
                reached = 0;  // T stays as it is
                n_above = reach.x;
            }
            if (reached == k) {  // exactly the candidates from T on
                --T;
                ties = 0;
                break;
            }
        }
        if (ties == 0 || shift < 0) break;
        const uint32_t width = 4u << shift;  // the undecided keys are T .. T + width - 1
        smallest = 0xffffffffu;
        largest = 0u;
        auto look_at = [&](uint32_t key) {
            if (key - T < width) {
                smallest = min(smallest, key);
                largest = max(largest, key);
            }
        };
#pragma unroll
        for (int e = 0; e < kSelectKeys; ++e)
            if (kSelectKeys > 8 || e < rounds) look_at(keys[e]);
        if (has_tail)
            for (int i = tail0 + tid; i < hi; i += kSelectThreads) look_at(select_key(score_at(i)));
    }
    if (ties < 0) ties = k - n_above;

    for (int i = tid; i < p.sink_blocks; i += kSelectThreads) idx[i] = i;
    for (int i = tid; i < p.local_blocks; i += kSelectThreads) idx[p.sink_blocks + k + i] = hi + i;
    // Ordered compaction (ascending block index = round e, then thread).  Register part: two ballots per round, the
    // (round, warp) counts scanned once by warp 0.
#pragma unroll
    for (int e = 0; e < kSelectKeys; ++e) {
        const bool in = lo + tid + e * kSelectThreads < hi;
        const unsigned above = __ballot_sync(0xffffffffu, in && keys[e] > T), tied = __ballot_sync(0xffffffffu, in && keys[e] == T);
        if (lane == 0) s_counts[e * kWarps + warp] = (unsigned)__popc(above) | (unsigned)__popc(tied) << 16;
    }
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the counts: some per lane, then across lanes
        constexpr int kEach = kCounts / 32;
        unsigned each[kEach], sum = 0;
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            each[u] = s_counts[lane * kEach + u];
            sum += each[u];
        }
        unsigned incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        unsigned run = incl - sum;
#pragma unroll
        for (int u = 0; u < kEach; ++u) {
            s_counts[lane * kEach + u] = run;
            run += each[u];
        }
        if (lane == 31) s_total = incl;
    }
    __syncthreads();
    const unsigned below_me = (1u << lane) - 1u;
    // candidate i: above T, or of key T; `above` and `tied` of either before it
    auto place = [&](int i, bool is_above, bool is_tied, int above, int tied) {
        if (is_above) idx[p.sink_blocks + above + min(tied, ties)] = i;
        if (is_tied && tied < ties) idx[p.sink_blocks + above + tied] = i;
    };
#pragma unroll
    for (int e = 0; e < kSelectKeys; ++e)
        if (e < rounds) {
            const bool in = lo + tid + e * kSelectThreads < hi, is_above = in && keys[e] > T, is_tied = in && keys[e] == T;
            const unsigned above = __ballot_sync(0xffffffffu, is_above), tied = __ballot_sync(0xffffffffu, is_tied);
            const unsigned before = s_counts[e * kWarps + warp];
            place(lo + tid + e * kSelectThreads, is_above, is_tied, (int)(before & 0xffffu) + __popc(above & below_me),
                  (int)(before >> 16) + __popc(tied & below_me));
        }
    if (!has_tail) return;
    // candidates beyond the register part: round by round
    int run_above = (int)(s_total & 0xffffu), run_tied = (int)(s_total >> 16);
    for (int base = tail0; base < hi; base += kSelectThreads) {
        const int i = base + tid;
        const uint32_t key = i < hi ? select_key(score_at(i)) : 0u;
        const bool is_above = i < hi && key > T, is_tied = i < hi && key == T;
        const unsigned above = __ballot_sync(0xffffffffu, is_above), tied = __ballot_sync(0xffffffffu, is_tied);
        __syncthreads();  // the counts of the previous round have been read by everyone
        if (lane == 0) s_counts[warp] = (unsigned)__popc(above) | (unsigned)__popc(tied) << 16;
        __syncthreads();
        unsigned before = 0, all = 0;
        for (int w = 0; w < kWarps; ++w) {
            if (w == warp) before = all;
            all += s_counts[w];
        }
        place(i, is_above, is_tied, run_above + (int)(before & 0xffffu) + __popc(above & below_me),
              run_tied + (int)(before >> 16) + __popc(tied & below_me));
        run_above += (int)(all & 0xffffu);
        run_tied += (int)(all >> 16);
    }
}

// ---------------------------------------------------------------------------------------------
// Gather: grid = (budget blocks, Hkv, layers x seqs); a CTA copies the valid tokens of one selected
// block's K and V (16-byte vectors) into the partial cache.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) gather_kernel(GatherParams p) {
    pdl_begin(p.pdl);
    const int s = blockIdx.x, h = blockIdx.y, lb = blockIdx.z;
    const int b = lb % p.batch, l = lb / p.batch;
    const int count = p.count[b];
    const int seq_len = p.seq_lens[b];
    const int nb = (seq_len + p.bs - 1) / p.bs;
    if (s == 0 && h == 0 && l == 0 && threadIdx.x == 0) {
        int plen = 0;
        // the last selected block is the sequence's last block (local window or, for short
        // contexts, simply every block): it keeps only its valid tokens
        if (count > 0) plen = (count - 1) * p.bs + (seq_len - (nb - 1) * p.bs);
        p.partial_lens[b] = plen;
    }
    if (s >= count) return;
    const int blk = p.idx[(((size_t)l * p.batch + b) * p.Hkv + h) * p.budget_blocks + s];
    if (blk < 0 || blk >= nb || blk >= p.full_max_blocks || s >= p.part_max_blocks) {
        if (threadIdx.x == 0) record_fault(p.workspace, SPECPV_ERR_INVALID_ARG, b, s, blk, l);
        return;
    }
    const int src_page = p.full_table[(size_t)b * p.full_max_blocks + blk];
    const int dst_page = p.part_table[(size_t)b * p.part_max_blocks + s];
    if (src_page < 0 || src_page >= p.full_pages || dst_page < 0 || dst_page >= p.part_pages) {
        if (threadIdx.x == 0) record_fault(p.workspace, SPECPV_ERR_BAD_BLOCK_TABLE, b, blk, src_page, dst_page);
        return;
    }
    const int n_valid = blk == nb - 1 ? seq_len - blk * p.bs : p.bs;
    const size_t row_bytes = (size_t)p.d * p.es;
    const size_t n_vec = (size_t)n_valid * row_bytes / 16;
    const size_t src_off = (((size_t)l * p.full_pages + src_page) * p.Hkv + h) * p.bs * row_bytes;
    const size_t dst_off = (((size_t)l * p.part_pages + dst_page) * p.Hkv + h) * p.bs * row_bytes;
    const uint4* ks = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(p.full_k) + src_off);
    const uint4* vs = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(p.full_v) + src_off);
    uint4* kd = reinterpret_cast<uint4*>(reinterpret_cast<char*>(p.part_k) + dst_off);
    uint4* vd = reinterpret_cast<uint4*>(reinterpret_cast<char*>(p.part_v) + dst_off);
    // up to four 16-byte loads of K and of V in flight per thread before the stores
    for (size_t i = threadIdx.x; i < n_vec; i += 4 * blockDim.x) {
        uint4 a[4], b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * blockDim.x < n_vec) {
                a[u] = ks[i + u * blockDim.x];
                b[u] = vs[i + u * blockDim.x];
            }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i + u * blockDim.x < n_vec) {
                kd[i + u * blockDim.x] = a[u];
                vd[i + u * blockDim.x] = b[u];
            }
    }
}

// ---------------------------------------------------------------------------------------------
// Commit: a CTA's four warps append the accepted tokens' K and V rows that fall into one block (a warp per row) and recompute the
// block's summary, the appended tokens taken from the step's tensors; grid = (blocks touched, KV heads, layers x seqs).  All CTAs
// read the lengths.  Up to four of them (one float32 layer, short steps) are one CTA that advances the lengths itself behind a barrier,
// up to eight one cluster that does so once they have all arrived; else the lengths advance in a launch behind them: a commit keeps
// nothing in the workspace but the status word, so that commits of two caches on two streams may share one (an arrival counter there
// made the launch unnecessary, 9.3 us a call against 11.4, but mixed the arrivals of two such commits).  Bound by launches.  us with a
// copy of the lengths, two launches / a CTA that took four units side by side and then the rest / cluster: four units of 4 tokens 6.1 /
// 6.5 / 5.8, eight 6.1 / 10.4 / 6.4 (a launch less for the host), eight of 46 tokens 10.1 / 18.1 / 10.0, of 64 16.7 / 31.9 / 16.5.  A cluster
// costs the host more: a float32 step with two commits of four units 65.3 us with clusters, 64.1 with a CTA.
// ---------------------------------------------------------------------------------------------
constexpr int kCommitWarps = 4;
constexpr int kCommitUnits = 4;    // of one CTA, side by side
constexpr int kCommitCluster = 8;  // CTAs of a cluster that every launch may ask for

template <typename T>
__device__ __forceinline__ void commit_unit(const CommitParams& p, int touched, int h, int lb, int warp, int lane) {
    const int b = lb % p.batch, l = lb / p.batch;
    const int n = min(max(p.n_accepted[b], 0), p.A_max);
    const int seq_len = p.seq_lens[b];
    const bool fits = (size_t)seq_len + n <= (size_t)p.max_blocks * p.bs;
    const int i = max(seq_len, 0) / p.bs + touched;  // logical block
    if (!fits) {
        if (warp == 0 && lane == 0 && touched == 0 && h == 0 && n > 0) record_fault(p.workspace, SPECPV_ERR_CAPACITY, b, seq_len, n, l);
    } else {
        const int t0 = max(seq_len, i * p.bs), t1 = min(seq_len + n, (i + 1) * p.bs);  // tokens appended to this block
        const bool summarise = p.kmax && (size_t)i * p.bs < (size_t)(seq_len + n) && i < p.max_blocks;
        int page = -1;
        if (t0 < t1 || summarise) {
            page = p.block_table[(size_t)b * p.max_blocks + i];
            if (page < 0 || page >= p.n_pages) {
                if (warp == 0 && lane == 0) record_fault(p.workspace, SPECPV_ERR_BAD_BLOCK_TABLE, b, i, page, l);
                page = -1;
            }
        }
        const int chunks = p.d * (int)sizeof(T) / 16;  // 16-byte chunks per row: 8, 16 or 32
        const size_t page0 = (((size_t)(p.layer0 + l) * p.n_pages + max(page, 0)) * p.Hkv + h) * p.bs;
        const uint4* k_new = reinterpret_cast<const uint4*>(p.k_new);
        const uint4* v_new = reinterpret_cast<const uint4*>(p.v_new);
        uint4* k_pool = reinterpret_cast<uint4*>(p.k_pool);
        uint4* v_pool = reinterpret_cast<uint4*>(p.v_pool);
        const int tok_lanes = 32 / chunks, chunk = lane % chunks, tl = lane / chunks;  // rows side by side in a warp
        // row of the step's tensors that token t takes, -1 if there is none
        auto source_row = [&](int t) {
            const int row = p.accepted[(size_t)b * p.A_max + t - seq_len];
            return row >= 0 && row < p.M_max ? row : -1;
        };
        if (page >= 0) {
            constexpr int kAhead = 4;  // rows in flight per lane
            const int step = kCommitWarps * tok_lanes;
            for (int t = t0 + warp * tok_lanes + tl; t < t1; t += kAhead * step) {
                uint4 kb[kAhead], vb[kAhead];
                int row[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    row[u] = t + u * step < t1 ? source_row(t + u * step) : -1;
                    if (row[u] >= 0) {
                        const size_t src = (((size_t)lb * p.M_max + row[u]) * p.Hkv + h) * chunks + chunk;
                        kb[u] = k_new[src];
                        vb[u] = v_new[src];
                    } else if (t + u * step < t1 && chunk == 0) {
                        const int a = t + u * step - seq_len;
                        record_fault(p.workspace, SPECPV_ERR_INVALID_ARG, b, a, p.accepted[(size_t)b * p.A_max + a], l);
                    }
                }
#pragma unroll
                for (int u = 0; u < kAhead; ++u)
                    if (row[u] >= 0) {
                        const size_t dst = (page0 + (t + u * step) % p.bs) * chunks + chunk;
                        k_pool[dst] = kb[u];
                        v_pool[dst] = vb[u];
                    }
            }
        }
        if (summarise && page >= 0 && warp == 0) {
            // as summaries_kernel, with the tokens of this commit read where they come from
            const int n_valid = min(p.bs, seq_len + n - i * p.bs);
            SummaryAcc<T> acc;
            for (int u0 = 0; u0 < n_valid; u0 += kSumLoads * tok_lanes) {
                uint4 buf[kSumLoads];
#pragma unroll
                for (int u = 0; u < kSumLoads; ++u) {
                    const int in = min(u0 + u * tok_lanes + tl, n_valid - 1), t = i * p.bs + in;
                    const uint4* src = k_pool + (page0 + in) * chunks;
                    if (t >= seq_len) {
                        const int row = source_row(t);
                        if (row >= 0) src = k_new + (((size_t)lb * p.M_max + row) * p.Hkv + h) * chunks;
                    }
                    buf[u] = src[chunk];
                }
#pragma unroll
                for (int u = 0; u < kSumLoads; ++u) acc.take(buf[u]);
            }
            acc.combine(chunks);
            if (tl == 0)
                acc.store(p.kmax, p.kmin, p.aligned,
                          ((((size_t)(p.layer0 + l) * p.batch + b) * p.Hkv + h) * p.max_blocks + i) * chunks + chunk);
        }
    }
}

__device__ __forceinline__ void advance_length(const CommitParams& p, int b) {
    const int n = min(max(p.n_accepted[b], 0), p.A_max);
    if ((size_t)p.seq_lens[b] + n <= (size_t)p.max_blocks * p.bs) p.seq_lens[b] += n;
}

template <typename T>
__global__ void __launch_bounds__(32 * kCommitWarps) commit_kernel(CommitParams p) {
    pdl_begin(p.pdl);
    commit_unit<T>(p, blockIdx.x, blockIdx.y, blockIdx.z, threadIdx.x >> 5, threadIdx.x & 31);
}

constexpr int kLensThreads = 128;
__global__ void __launch_bounds__(kLensThreads) commit_lens_kernel(CommitParams p) {
    pdl_begin(p.pdl);
    const int b = blockIdx.x * kLensThreads + threadIdx.x;
    if (b < p.batch) advance_length(p, b);
}

// One CTA for up to kCommitUnits units side by side, which advances the lengths itself behind a barrier.
template <typename T>
__global__ void __launch_bounds__(32 * kCommitWarps * kCommitUnits) commit_small_kernel(CommitParams p, dim3 units) {
    pdl_begin(1);
    const int u = threadIdx.x / (32 * kCommitWarps);
    if (u < (int)(units.x * units.y * units.z))
        commit_unit<T>(p, u % units.x, u / units.x % units.y, u / (units.x * units.y), (threadIdx.x >> 5) % kCommitWarps, threadIdx.x & 31);
    __syncthreads();  // every unit has read the lengths
    if ((int)threadIdx.x < p.batch) advance_length(p, threadIdx.x);
}

// One cluster, a CTA per unit, which advances the lengths itself.
template <typename T>
__global__ void __launch_bounds__(32 * kCommitWarps) commit_cluster_kernel(CommitParams p) {
    pdl_begin(1);
    commit_unit<T>(p, blockIdx.x, blockIdx.y, blockIdx.z, threadIdx.x >> 5, threadIdx.x & 31);
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");  // every unit has read the lengths
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && (int)threadIdx.x < p.batch) advance_length(p, threadIdx.x);
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------------
#define SPECPV_LAUNCH(...)                                                     \
    do {                                                                       \
        if (launch_pdl_if(__VA_ARGS__) != cudaSuccess) return SPECPV_ERR_CUDA; \
        count_launch();                                                        \
    } while (0)

specpv_status launch_summaries(const SummaryParams& params, int n_layers, int blocks_touched, int dtype,
                               cudaStream_t stream) {
    if (blocks_touched <= 0 || n_layers <= 0) return SPECPV_OK;
    SummaryParams p = params;
    p.aligned = aligned16(p.kmax) && aligned16(p.kmin);
    const int warps = p.Hkv < kSumWarps ? p.Hkv : kSumWarps;
    dim3 grid(blocks_touched, (p.Hkv + kSumWarps - 1) / kSumWarps, n_layers * p.batch);
    SPECPV_LAUNCH(dtype == SPECPV_DTYPE_F32 ? summaries_kernel<float> : summaries_kernel<__nv_bfloat16>, grid, 32 * warps, 0, stream, p);
    return SPECPV_OK;
}

template <typename T, int D, int kBlocks, int kParts>
static specpv_status launch_scores_form(const ScoreParams& p, int n_layers, int max_nb, cudaStream_t stream) {
    constexpr int kCtaBlocks = kScoreWarps * kBlocks;
    const size_t smem = (size_t)((kParts == 1 ? kScoreRows : kScoreFewRows) * (D + 4) + kCtaBlocks * 2 * D) * sizeof(float);
    if (!tc::set_smem_limit_once(reinterpret_cast<const void*>(scores_simt_kernel<T, D, kBlocks, kParts>), (int)smem)) return SPECPV_ERR_CUDA;
    dim3 grid((max_nb + kCtaBlocks - 1) / kCtaBlocks, p.Hkv, n_layers * p.batch);
    SPECPV_LAUNCH((scores_simt_kernel<T, D, kBlocks, kParts>), grid, 32 * kScoreWarps, smem, stream, p);
    return SPECPV_OK;
}

template <typename T, int D>
static specpv_status launch_scores_typed(const ScoreParams& p, int n_layers, int max_nb, cudaStream_t stream) {
    // four blocks per warp once that still gives two CTAs to every SM
    const long long ctas = (long long)((max_nb + 4 * kScoreWarps - 1) / (4 * kScoreWarps)) * p.Hkv * n_layers * p.batch;
    const bool four = ctas >= 2 * 148;
    // eight lanes to a row up to 16 rows, with one block per warp up to 8 (16 rows of 64, 128 blocks x 8 lists: 3.35 -> 3.65 us with them)
    const int rows = p.reduce == SPECPV_REDUCE_LAST ? p.G : p.M_max * p.G;
    if (four)
        return rows <= kScoreFewRows ? launch_scores_form<T, D, 4, 8>(p, n_layers, max_nb, stream) : launch_scores_form<T, D, 4, 1>(p, n_layers, max_nb, stream);
    return rows <= kScoreFewRows / 2 ? launch_scores_form<T, D, 1, 8>(p, n_layers, max_nb, stream) : launch_scores_form<T, D, 1, 1>(p, n_layers, max_nb, stream);
}

specpv_status launch_scores(const ScoreParams& p, int n_layers, int max_nb, int dtype, int d, cudaStream_t stream) {
    if (max_nb <= 0 || n_layers <= 0) return SPECPV_OK;
    if (dtype == SPECPV_DTYPE_F32) {
        if (d == 64) return launch_scores_typed<float, 64>(p, n_layers, max_nb, stream);
        if (d == 128) return launch_scores_typed<float, 128>(p, n_layers, max_nb, stream);
    } else {
        if (d == 64) return launch_scores_typed<__nv_bfloat16, 64>(p, n_layers, max_nb, stream);
        if (d == 128) return launch_scores_typed<__nv_bfloat16, 128>(p, n_layers, max_nb, stream);
    }
    return SPECPV_ERR_SHAPE;
}

specpv_status launch_select(const SelectParams& p, int n_layers, cudaStream_t stream) {
    if (n_layers <= 0 || p.batch <= 0) return SPECPV_OK;
    const dim3 grid(p.Hkv, p.batch, n_layers);
    // By the most candidates a list can have; up to a list per SM, twice the threads with half the keys each (3837 x 128: 13.0 -> 10.4 us,
    // 8189 x 8: 16.7 -> 14.6, both with more code), above that they only crowd (4090 x 256: 15.6 -> 21.0).
    const int n = p.max_blocks - p.sink_blocks - p.local_blocks;
    const bool few = (long long)grid.x * grid.y * grid.z <= 148;
    if (n <= 1024)
        SPECPV_LAUNCH((select_kernel<256, 4>), grid, 256, 0, stream, p);
    else if (n <= 2048)
        SPECPV_LAUNCH((select_kernel<512, 4>), grid, 512, 0, stream, p);
    else if (n <= 4096 && few)
        SPECPV_LAUNCH((select_kernel<1024, 4>), grid, 1024, 0, stream, p);
    else if (n <= 4096)
        SPECPV_LAUNCH((select_kernel<512, 8>), grid, 512, 0, stream, p);
    else if (n <= 8192 && few)
        SPECPV_LAUNCH((select_kernel<1024, 8>), grid, 1024, 0, stream, p);
    else if (n <= 8192)
        SPECPV_LAUNCH((select_kernel<512, 16>), grid, 512, 0, stream, p);
    else
        SPECPV_LAUNCH((select_kernel<1024, 16, true>), grid, 1024, 0, stream, p);
    return SPECPV_OK;
}

specpv_status launch_gather(const GatherParams& p, int n_layers, cudaStream_t stream) {
    dim3 grid(p.budget_blocks, p.Hkv, n_layers * p.batch);
    SPECPV_LAUNCH(gather_kernel, grid, 128, 0, stream, p);
    return SPECPV_OK;
}

specpv_status launch_commit(const CommitParams& params, int n_layers, int dtype, bool advance, cudaStream_t stream) {
    CommitParams p = params;
    p.aligned = aligned16(p.kmax) && aligned16(p.kmin);
    dim3 grid((p.A_max + p.bs - 1) / p.bs + 1, p.Hkv, n_layers * p.batch);
    const long long units = (long long)grid.x * grid.y * grid.z;
    if (advance && units <= kCommitUnits) {
        if (launch_pdl(dtype == SPECPV_DTYPE_F32 ? commit_small_kernel<float> : commit_small_kernel<__nv_bfloat16>, 1,
                       32 * kCommitWarps * (int)units, 0, stream, p, grid) != cudaSuccess)
            return SPECPV_ERR_CUDA;
        count_launch();
        return SPECPV_OK;
    }
    if (advance && units <= kCommitCluster) {
        cudaLaunchAttribute attr[2]{};
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = grid.x;
        attr[1].val.clusterDim.y = grid.y;
        attr[1].val.clusterDim.z = grid.z;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = grid;
        cfg.blockDim = 32 * kCommitWarps;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
        if (cudaLaunchKernelEx(&cfg, dtype == SPECPV_DTYPE_F32 ? commit_cluster_kernel<float> : commit_cluster_kernel<__nv_bfloat16>, p) != cudaSuccess)
            return SPECPV_ERR_CUDA;
        count_launch();
        return SPECPV_OK;
    }
    SPECPV_LAUNCH(dtype == SPECPV_DTYPE_F32 ? commit_kernel<float> : commit_kernel<__nv_bfloat16>, grid, 32 * kCommitWarps, 0, stream, p);
    if (advance) SPECPV_LAUNCH(commit_lens_kernel, dim3((p.batch + kLensThreads - 1) / kLensThreads), kLensThreads, 0, stream, p);
    return SPECPV_OK;
}

}  // namespace specpv
