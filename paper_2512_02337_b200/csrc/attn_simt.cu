// Tree-masked GQA verification attention, float32 SIMT path (paper Section 3.2-3.3, Algorithm 1
// "TreeDecode").  Covers every geometry (float32 or bfloat16 storage, any group size, any block
// size) with float32 arithmetic and accurate expf; it is the path for float32 caches and the
// on-device second opinion for the tensor-core kernel.
//
// Work split: one CTA per (layer, sequence, KV head, KV split, tile of 64 query rows).  A CTA walks its share of the
// 64-token tiles (the tiles of the step's own tokens come last, under the tree mask): Q, K and V are staged in shared memory
// as float32 (Q and K channel-major), a thread owns four rows and four tokens of S and four rows and D/16 channels of O, so
// both products are register-tiled, and the running (max, sum, accumulator) of the online softmax stay in registers.
// With more than one split the unnormalised partial results go to the workspace and merge_splits_kernel combines them with
// a log-sum-exp merge.
// Short calls are bound by latency: the form before this one (a warp per four rows, a lane per token, 256 tokens per CTA)
// left a 2048-token call on 16 CTAs.  8 query heads of 64, 2 KV heads, 16 rows, float32: 2048 tokens 119 -> 18 us.
// Larger ones are bound by shared-memory reads, two 16-byte loads per 16 multiplications, which are done in packed pairs (32 rows,
// 8192 tokens x 4 layers: 283 -> 108 us, one layer at a time 28.8 -> 26.7 by the packing).
#include <math.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace specpv {

namespace {

constexpr int kThreads = 256;
constexpr int kTok = 64;          // tokens per tile
constexpr int kRows = 64;         // query rows per CTA
constexpr int kPitch = kTok + 4;  // row pitch of the staged tiles (keeps float4 alignment)

// dynamic shared memory: Q [D][kPitch], K [D][kPitch] (both channel-major), V [kTok][D], P [kRows][kPitch]
template <int D>
constexpr size_t simt_smem() {
    return (size_t)(2 * D * kPitch + kTok * D + kRows * kPitch) * sizeof(float);
}

struct SimtParams {
    const void* q;
    const void* k_new;
    const void* v_new;
    const uint64_t* tree_mask;
    const int32_t* q_lens;
    const void* k_pool;
    const void* v_pool;
    const int32_t* block_table;
    const int32_t* seq_lens;
    void* out;
    float* lse;
    float* part_o;   // [lb][Hkv][splits][R_max][D]
    float* part_ml;  // [lb][Hkv][splits][R_max][2]
    void* workspace;
    int layer0, batch, M_max, mask_words, Hq, Hkv, G, bs, max_blocks, n_pages;
    int n_splits, row_tiles;
    int pdl;  // set by launch_pdl_if
    float scale;
};

// reductions over the 16 lanes that share a row
__device__ __forceinline__ float row_max(float v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float row_sum(float v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// four consecutive values as float32 (16-byte aligned for float32, 8-byte for bfloat16)
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xFFFF0000u));
}

template <typename T, typename TO, int D>
__global__ void __launch_bounds__(kThreads) attn_simt_kernel(SimtParams p) {
    pdl_begin(p.pdl);
    constexpr int CPT = D / 16;   // output channels per thread
    constexpr int kLoads = D / 16;  // float4 loads per thread of a 64 x D tile
    extern __shared__ float smem[];
    float* Qt = smem;
    float* Kt = Qt + D * kPitch;
    float* Vs = Kt + D * kPitch;
    float* Ps = Vs + kTok * D;
    __shared__ uint64_t s_mask[kRows][2];  // step tokens each row sees
    __shared__ __align__(4) unsigned char s_exists[kTok];  // whether the tile has this token (one behind a bad page id is skipped)

    const int split = blockIdx.x % p.n_splits, row0 = blockIdx.x / p.n_splits * kRows;
    const int h = blockIdx.y, lb = blockIdx.z;
    const int b = lb % p.batch, l = lb / p.batch;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const int seq_len = max(p.seq_lens[b], 0);
    int M = p.q_lens ? p.q_lens[b] : p.M_max;
    M = min(max(M, 0), p.M_max);
    const int R = M * p.G, R_max = p.M_max * p.G;
    if (row0 >= R) return;

    const int ctx_tiles = (seq_len + kTok - 1) / kTok, positions = ctx_tiles + (M + kTok - 1) / kTok;
    const int tile_begin = (int)((long long)positions * split / p.n_splits);
    const int tile_end = (int)((long long)positions * (split + 1) / p.n_splits);

    const T* q = reinterpret_cast<const T*>(p.q) + (size_t)lb * p.M_max * p.Hq * D;
    const T* k_new = reinterpret_cast<const T*>(p.k_new) + (size_t)lb * p.M_max * p.Hkv * D;
    const T* v_new = reinterpret_cast<const T*>(p.v_new) + (size_t)lb * p.M_max * p.Hkv * D;
    const size_t layer_stride = (size_t)p.n_pages * p.Hkv * p.bs * D;
    const T* k_pool = reinterpret_cast<const T*>(p.k_pool) + (size_t)(p.layer0 + l) * layer_stride;
    const T* v_pool = reinterpret_cast<const T*>(p.v_pool) + (size_t)(p.layer0 + l) * layer_stride;
    const int32_t* table = p.block_table + (size_t)b * p.max_blocks;
    const uint64_t* mask = p.tree_mask + (size_t)b * p.M_max * p.mask_words;

    // staging: a thread takes row or token tid % 64, and of it the 16-byte pieces tid / 64, + 4, ..
    const int st = tid % kTok, sc = tid / kTok;
    {
        const int r = row0 + st;
        const T* src = q + ((size_t)(r / p.G) * p.Hq + h * p.G + r % p.G) * D;
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int c = (sc + 4 * i) * 4;
            const float4 v = r < R ? load4(src + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            Qt[(c + 0) * kPitch + st] = v.x;
            Qt[(c + 1) * kPitch + st] = v.y;
            Qt[(c + 2) * kPitch + st] = v.z;
            Qt[(c + 3) * kPitch + st] = v.w;
        }
        if (tid < kRows) {
            const uint64_t* m = mask + (size_t)(r / p.G) * p.mask_words;
            s_mask[tid][0] = r < R ? m[0] : 0ull;
            s_mask[tid][1] = r < R && p.mask_words > 1 ? m[1] : 0ull;
        }
    }
    // K and V rows of tile `tile` for this thread's token, in flight while the previous tile is worked on
    float4 kbuf[kLoads], vbuf[kLoads];
    bool exists = false;
    auto fetch = [&](int tile) {
        const T *ks = nullptr, *vs = nullptr;
        if (tile < ctx_tiles) {
            const int t = tile * kTok + st;
            if (t < seq_len) {
                const int page = table[t / p.bs];
                if (page >= 0 && page < p.n_pages) {
                    const size_t off = (((size_t)page * p.Hkv + h) * p.bs + t % p.bs) * D;
                    ks = k_pool + off;
                    vs = v_pool + off;
                } else if (sc == 0 && row0 == 0) {
                    record_fault(p.workspace, SPECPV_ERR_BAD_BLOCK_TABLE, b, t / p.bs, page, l);
                }
            }
        } else if ((tile - ctx_tiles) * kTok + st < M) {
            const size_t off = ((size_t)((tile - ctx_tiles) * kTok + st) * p.Hkv + h) * D;
            ks = k_new + off;
            vs = v_new + off;
        }
        exists = ks != nullptr;
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int c = (sc + 4 * i) * 4;
            kbuf[i] = ks ? load4(ks + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            vbuf[i] = vs ? load4(vs + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float m_run[4], l_run[4], acc[4][CPT];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m_run[i] = -INFINITY;
        l_run[i] = 0.f;
#pragma unroll
        for (int c = 0; c < CPT; ++c) acc[i][c] = 0.f;
    }
    if (tile_begin < tile_end) fetch(tile_begin);
    for (int tile = tile_begin; tile < tile_end; ++tile) {
        const bool is_new = tile >= ctx_tiles;
        const int tok0 = (is_new ? tile - ctx_tiles : tile) * kTok;
        __syncthreads();  // the previous tile has been read
#pragma unroll
        for (int i = 0; i < kLoads; ++i) {
            const int c = (sc + 4 * i) * 4;
            Kt[(c + 0) * kPitch + st] = kbuf[i].x;
            Kt[(c + 1) * kPitch + st] = kbuf[i].y;
            Kt[(c + 2) * kPitch + st] = kbuf[i].z;
            Kt[(c + 3) * kPitch + st] = kbuf[i].w;
            *reinterpret_cast<float4*>(Vs + st * D + c) = vbuf[i];
        }
        if (sc == 0) s_exists[st] = exists;
        __syncthreads();
        if (tile + 1 < tile_end) fetch(tile + 1);
        // S = Q K^T: rows 4 ty .. + 3, tokens 4 tx .. + 3.  Channels are summed in runs of 16, the runs then added: the
        // rounding of a long serial sum would show in the weights of the largest logits.
        float2 sp[4][2];  // tokens (0, 1) and (2, 3)
#pragma unroll
        for (int i = 0; i < 4; ++i) sp[i][0] = sp[i][1] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 16) {
            float2 part[4][2];
#pragma unroll
            for (int cc = 0; cc < 16; ++cc) {
                const float4 a = *reinterpret_cast<const float4*>(Qt + (c0 + cc) * kPitch + 4 * ty);
                const float4 k4 = *reinterpret_cast<const float4*>(Kt + (c0 + cc) * kPitch + 4 * tx);
                const float av[4] = {a.x, a.y, a.z, a.w};
                const float2 kv[2] = {make_float2(k4.x, k4.y), make_float2(k4.z, k4.w)};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        part[i][j] = cc == 0 ? __fmul2_rn(make_float2(av[i], av[i]), kv[j]) : __ffma2_rn(make_float2(av[i], av[i]), kv[j], part[i][j]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) sp[i][j] = __fadd2_rn(sp[i][j], part[i][j]);
        }
        float sv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sv[i][0] = sp[i][0].x; sv[i][1] = sp[i][0].y; sv[i][2] = sp[i][1].x; sv[i][3] = sp[i][1].y;
        }
        const uchar4 e4 = *reinterpret_cast<const uchar4*>(s_exists + 4 * tx);
        const unsigned in_tile = (unsigned)e4.x | (unsigned)e4.y << 1 | (unsigned)e4.z << 2 | (unsigned)e4.w << 3;
        float corr[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            unsigned vis = in_tile;
            if (is_new) vis &= (unsigned)(s_mask[4 * ty + i][(tok0 + 4 * tx) >> 6] >> ((4 * tx) & 63)) & 15u;
            float mx = -INFINITY;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sv[i][j] = (vis >> j) & 1u ? sv[i][j] * p.scale : -INFINITY;
                mx = fmaxf(mx, sv[i][j]);
            }
            const float m_new = fmaxf(m_run[i], row_max(mx));
            const float m_safe = m_new == -INFINITY ? 0.f : m_new;
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sv[i][j] = expf(sv[i][j] - m_safe);  // exp(-inf) = 0 for masked keys
                sum += sv[i][j];
            }
            corr[i] = expf(m_run[i] - m_safe);  // 0 while nothing has been seen
            l_run[i] = l_run[i] * corr[i] + row_sum(sum);
            m_run[i] = m_new;
            *reinterpret_cast<float4*>(Ps + (4 * ty + i) * kPitch + 4 * tx) = make_float4(sv[i][0], sv[i][1], sv[i][2], sv[i][3]);
        }
        __syncwarp();  // the rows a thread reads below were written by its own half warp
        // O = O corr + P V, channels c * 16 + 4 tx + ..: the tile's 64 products are summed apart and then added, because one chain
        // over a CTA's whole share (2112 tokens of 8192 with 240 rows x 8 heads x 2 layers) loses digits (8.9e-7 against 8.2e-7
        // with 432 tokens to a chain).
        float2 tile_acc[4][CPT / 2];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < CPT / 2; ++c) tile_acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int t = 0; t < kTok; t += 4) {
            float4 pr[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) pr[i] = *reinterpret_cast<const float4*>(Ps + (4 * ty + i) * kPitch + t);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float2 vv[CPT / 2];
#pragma unroll
                for (int c = 0; c < CPT; c += 4) {
                    const float4 v4 = *reinterpret_cast<const float4*>(Vs + (t + u) * D + c * 16 + 4 * tx);
                    vv[c / 2] = make_float2(v4.x, v4.y);
                    vv[c / 2 + 1] = make_float2(v4.z, v4.w);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float w = u == 0 ? pr[i].x : u == 1 ? pr[i].y : u == 2 ? pr[i].z : pr[i].w;
#pragma unroll
                    for (int c = 0; c < CPT / 2; ++c) tile_acc[i][c] = __ffma2_rn(make_float2(w, w), vv[c], tile_acc[i][c]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < CPT; ++c) acc[i][c] = fmaf(acc[i][c], corr[i], c % 2 ? tile_acc[i][c / 2].y : tile_acc[i][c / 2].x);
    }
    // acc[i][c .. c + 3] are channels 16 c + 4 tx .. + 3 of row 4 ty + i
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = row0 + 4 * ty + i;
        if (r >= R) continue;
        if (p.n_splits == 1) {
            const int j = r / p.G, g = r % p.G;
            const size_t row = ((size_t)lb * p.M_max + j) * p.Hq + h * p.G + g;
            TO* o = reinterpret_cast<TO*>(p.out) + row * D;
            const float inv = 1.f / l_run[i];
#pragma unroll
            for (int c = 0; c < CPT; ++c) o[c / 4 * 64 + 4 * tx + c % 4] = from_float<TO>(acc[i][c] * inv);
            if (p.lse && tx == 0) p.lse[row] = m_run[i] + logf(l_run[i]);
        } else {
            const size_t prow = (((size_t)lb * p.Hkv + h) * p.n_splits + split) * R_max + r;
#pragma unroll
            for (int c = 0; c < CPT; c += 4)
                *reinterpret_cast<float4*>(p.part_o + prow * D + c / 4 * 64 + 4 * tx) =
                    make_float4(acc[i][c], acc[i][c + 1], acc[i][c + 2], acc[i][c + 3]);
            if (tx == 0) {
                p.part_ml[prow * 2] = m_run[i];
                p.part_ml[prow * 2 + 1] = l_run[i];
            }
        }
    }
}

// Log-sum-exp merge of the per-split partial results: D/4 threads per row and group of D/4 splits, four channels each, eight
// partial rows in flight per thread; a row's groups (up to 64 splits in all) meet in shared memory and are added in order.  Bound by
// latency: 64 splits one group of lanes after the other took 8.1 us a call, side by side 4.6; 33 splits 5.9 and 3.5.  Fewer splits, where groups
// idle, with the attention before the merge (64 rows of 64 channels): 2 splits 12.2 -> 11.0 us, 5 12.4 -> 11.0, 9 12.8 -> 11.6.
// grid = (row groups, KV heads, layers x seqs).
constexpr int kMergeThreads = 128;
constexpr int kMergeAhead = 8;
template <typename TO, int D>
__global__ void __launch_bounds__(kMergeThreads) merge_splits_kernel(SimtParams p) {
    pdl_begin(p.pdl);
    constexpr int kRowThreads = D / 4, kGroups = 64 / kRowThreads, kRowsAtOnce = kMergeThreads / 64;
    __shared__ float4 s_o[kMergeThreads];
    __shared__ float s_l[kMergeThreads];
    const int r = blockIdx.x * kRowsAtOnce + threadIdx.x / 64;
    const int h = blockIdx.y, lb = blockIdx.z, lane = threadIdx.x % kRowThreads, group = threadIdx.x % 64 / kRowThreads;
    const int b = lb % p.batch;
    int M = p.q_lens ? p.q_lens[b] : p.M_max;
    M = min(max(M, 0), p.M_max);
    const bool row_valid = r < M * p.G;
    const unsigned members = kRowThreads == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
    const int R_max = p.M_max * p.G;
    const size_t row0 = ((size_t)lb * p.Hkv + h) * p.n_splits * R_max + (row_valid ? r : 0);
    const int c0 = group * kRowThreads, n = min(kRowThreads, p.n_splits - c0);  // this group's splits
    const float4* po = reinterpret_cast<const float4*>(p.part_o + row0 * D) + lane;
    const float2* ml = reinterpret_cast<const float2*>(p.part_ml) + row0;
    const size_t po_stride = (size_t)R_max * kRowThreads;
    float4 buf[kMergeAhead];
    auto fetch = [&](int s0) {
#pragma unroll
        for (int u = 0; u < kMergeAhead; ++u)
            if (s0 + u < n) buf[u] = po[(size_t)(c0 + s0 + u) * po_stride];
    };
    fetch(0);
    float m_all = -INFINITY;
    float2 mine = make_float2(-INFINITY, 0.f);  // of split c0 + lane
#pragma unroll
    for (int g = 0; g < kGroups; ++g)
        if (g * kRowThreads + lane < p.n_splits) {
            const float2 v = ml[(size_t)(g * kRowThreads + lane) * R_max];
            m_all = fmaxf(m_all, v.x);
            if (g == group) mine = v;
        }
#pragma unroll
    for (int o = kRowThreads / 2; o > 0; o >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(members, m_all, o));
    float w_mine = 0.f, l_mine = 0.f;
    if (mine.x != -INFINITY) {  // a split that saw no token weighs nothing
        w_mine = expf(mine.x - m_all);
        l_mine = mine.y * w_mine;
    }
    float l_all = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < n; s0 += kMergeAhead) {
        if (s0) fetch(s0);
#pragma unroll
        for (int u = 0; u < kMergeAhead; ++u) {  // (D/4 is a multiple of kMergeAhead: the shuffles stay among the row's lanes)
            const float w = __shfl_sync(members, w_mine, s0 + u, kRowThreads);
            const float lw = __shfl_sync(members, l_mine, s0 + u, kRowThreads);
            if (s0 + u >= n || w == 0.f) continue;
            l_all += lw;
            o.x = fmaf(buf[u].x, w, o.x);
            o.y = fmaf(buf[u].y, w, o.y);
            o.z = fmaf(buf[u].z, w, o.z);
            o.w = fmaf(buf[u].w, w, o.w);
        }
    }
    s_o[threadIdx.x] = o;
    s_l[threadIdx.x] = l_all;
    __syncthreads();
    if (!row_valid || group) return;
#pragma unroll
    for (int g = 1; g < kGroups; ++g) {
        if (g * kRowThreads >= p.n_splits) break;
        const float4 v = s_o[threadIdx.x + g * kRowThreads];
        o.x += v.x; o.y += v.y; o.z += v.z; o.w += v.w;
        l_all += s_l[threadIdx.x + g * kRowThreads];
    }
    const int j = r / p.G, g = r % p.G;
    const size_t row = ((size_t)lb * p.M_max + j) * p.Hq + h * p.G + g;
    TO* dst = reinterpret_cast<TO*>(p.out) + row * D + lane * 4;
    const float inv = 1.f / l_all;
    dst[0] = from_float<TO>(o.x * inv);
    dst[1] = from_float<TO>(o.y * inv);
    dst[2] = from_float<TO>(o.z * inv);
    dst[3] = from_float<TO>(o.w * inv);
    if (p.lse && lane == 0) p.lse[row] = m_all + logf(l_all);
}

template <typename T, typename TO, int D>
specpv_status launch_typed(const AttnArgs& a, SimtParams& p, cudaStream_t stream) {
    constexpr size_t smem = simt_smem<D>();
    if (!tc::set_smem_limit_once(reinterpret_cast<const void*>(attn_simt_kernel<T, TO, D>), (int)smem)) return SPECPV_ERR_CUDA;
    dim3 grid(p.n_splits * p.row_tiles, a.g.Hkv, a.n_layers * a.batch);
    if (launch_pdl_if(attn_simt_kernel<T, TO, D>, grid, kThreads, smem, stream, p) != cudaSuccess) return SPECPV_ERR_CUDA;
    count_launch();
    if (p.n_splits > 1) {
        constexpr int rows = kMergeThreads / 64;
        dim3 mgrid((a.M_max * a.g.G + rows - 1) / rows, a.g.Hkv, a.n_layers * a.batch);
        if (launch_pdl_if(merge_splits_kernel<TO, D>, mgrid, kMergeThreads, 0, stream, p) != cudaSuccess) return SPECPV_ERR_CUDA;
        count_launch();
    }
    return SPECPV_OK;
}

}  // namespace

specpv_status launch_attention_simt(const AttnArgs& a, cudaStream_t stream) {
    SimtParams p{};
    p.q = a.q; p.k_new = a.k_new; p.v_new = a.v_new; p.tree_mask = a.tree_mask; p.q_lens = a.q_lens;
    p.k_pool = a.k_pool; p.v_pool = a.v_pool; p.block_table = a.block_table; p.seq_lens = a.seq_lens;
    p.out = a.out; p.lse = a.lse; p.workspace = a.workspace;
    p.layer0 = a.layer0; p.batch = a.batch; p.M_max = a.M_max; p.mask_words = a.mask_words;
    p.Hq = a.g.Hq; p.Hkv = a.g.Hkv; p.G = a.g.G; p.bs = a.g.bs; p.max_blocks = a.max_blocks; p.n_pages = a.n_pages;
    p.scale = a.g.scale;

    // split the KV range so that the launch has up to 296 CTAs, down to one tile per CTA (a tile takes some 3 us, a partial result a
    // fraction of one), as far as the workspace allows: two CTAs per SM with 64 channels; with 128, where shared memory
    // holds one, two waves
    constexpr int kTargetCtas = 2 * 148;
    const int base = a.g.Hkv * a.n_layers * a.batch;
    const int R_max = a.M_max * a.g.G;
    p.row_tiles = (R_max + kRows - 1) / kRows;
    const int positions = (a.max_seq_len + kTok - 1) / kTok + (a.M_max + kTok - 1) / kTok;
    int n_splits = kTargetCtas / (base * p.row_tiles);
    if (n_splits > positions) n_splits = positions;
    if (n_splits > 64) n_splits = 64;
    const size_t per_split = (size_t)base * R_max * (a.g.d + 2) * sizeof(float);
    if (n_splits > 1 && per_split * n_splits > a.partial_bytes) n_splits = (int)(a.partial_bytes / per_split);
    if (n_splits < 1) n_splits = 1;
    p.n_splits = n_splits;
    char* ws = reinterpret_cast<char*>(a.workspace) + a.partial_off;
    p.part_o = reinterpret_cast<float*>(ws);
    p.part_ml = reinterpret_cast<float*>(ws + (size_t)base * n_splits * R_max * a.g.d * sizeof(float));

    if (a.g.dtype == SPECPV_DTYPE_F32) {
        if (a.g.d == 64) return launch_typed<float, float, 64>(a, p, stream);
        if (a.g.d == 128) return launch_typed<float, float, 128>(a, p, stream);
    } else if (a.g.out_f32) {
        if (a.g.d == 64) return launch_typed<__nv_bfloat16, float, 64>(a, p, stream);
        if (a.g.d == 128) return launch_typed<__nv_bfloat16, float, 128>(a, p, stream);
    } else {
        if (a.g.d == 64) return launch_typed<__nv_bfloat16, __nv_bfloat16, 64>(a, p, stream);
        if (a.g.d == 128) return launch_typed<__nv_bfloat16, __nv_bfloat16, 128>(a, p, stream);
    }
    return SPECPV_ERR_SHAPE;
}

}  // namespace specpv
