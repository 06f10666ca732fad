// Shared declarations of the SpecPV CUDA library: validated geometry, the device status word,
// workspace carving and dtype helpers.  Nothing here is shared with the CPU oracle.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/specpv.h"

namespace specpv {

// ---- device status word: workspace[0..255] ------------------------------------------------
// word 0: first recorded specpv_status (0 = none); words 1..4: details of that first fault.
struct StatusWord {
    int32_t code;
    int32_t info[4];
};

__device__ __forceinline__ void record_fault(void* workspace, int code, int i0, int i1, int i2, int i3) {
    StatusWord* sw = reinterpret_cast<StatusWord*>(workspace);
    if (atomicCAS(&sw->code, 0, code) == 0) {
        sw->info[0] = i0;
        sw->info[1] = i1;
        sw->info[2] = i2;
        sw->info[3] = i3;
    }
}

constexpr size_t kStatusBytes = 256;
// Head of every workspace: the status word, then arrival counters of KV ranges shared between CTAs (two per (layer,
// sequence, KV head, group of 256 rows) of a call; zero between launches).  All scratch starts behind it.
constexpr size_t kHeaderBytes = 256 * 1024;
constexpr int kMaxQTokens = 128;      // M_max supported by the attention kernels (two mask words)
constexpr int kMaxSplitCtas = 8 * 148;  // the workspace holds split-KV partial results of this many CTAs (+ one per head)

// ---- programmatic dependent launch ---------------------------------------------------------------
// Kernels are launched so that the next one on the stream may become resident while this one still runs (once every CTA of
// this one has called pdl_trigger() or ended): its launch and set-up hide behind this kernel's tail.  pdl_wait() returns when
// all earlier work on the stream is complete and visible; every kernel calls it before it reads or writes anything in
// global memory that a call passes in (L2 prefetches excepted), so the results are those of plain stream order.  A kernel
// that holds tensor memory triggers after it has allocated it: a later kernel's allocation can only wait for one that is
// already held, never the other way round.  While such a kernel runs, its predecessor may still be writing what it will read: it uses
// plain loads behind pdl_wait(), never loads through the read-only path (__ldg, const __restrict__ parameters), which are promised
// memory that nobody writes during the kernel and which the compiler may move ahead of the wait.  The attention kernel triggers when it has written its partial results: merge
// CTAs let in earlier pile up on the few SMs that it leaves free and run there one behind the other (one layer, 4096 tokens:
// 18.5 us against 16.8).  One layer's QKV projection, partial verification and output projection: 49.1 -> 43.7 us at a
// 4096-token budget, 43.7 -> 38.0 us at 2048.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The wait costs every CTA a few hundred nanoseconds, so a kernel of many short CTAs is launched the ordinary way (block
// summaries of 96K tokens x 32 layers, 49152 CTAs: 1040 us with it, 940 without); such kernels take the flag in their
// parameters (launch_pdl_if).  Kernels whose CTAs run for many microseconds (attention, block scores, projections) and the rope
// table, a CTA per row of a step, are always launched as dependents.
constexpr long long kPdlMaxCtas = 8 * 148;
inline bool pdl_pays(dim3 grid) { return (long long)grid.x * grid.y * grid.z <= kPdlMaxCtas; }
__device__ __forceinline__ void pdl_begin(int on) {
    if (on) {
        pdl_trigger();
        pdl_wait();
    }
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_plain(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const Args&... args) {
    kernel<<<grid, block, smem, stream>>>(KArgs(args)...);
    return cudaGetLastError();
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const Args&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
// for kernels whose parameter block says whether to wait
template <typename Params>
inline cudaError_t launch_pdl_if(void (*kernel)(Params), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Params p) {
    p.pdl = pdl_pays(grid);
    return p.pdl ? launch_pdl(kernel, grid, block, smem, stream, p) : launch_plain(kernel, grid, block, smem, stream, p);
}

// process-wide count of kernel launches (reported by specpv_kernel_launches)
void count_launch(int n = 1);

// ---- geometry after validation ---------------------------------------------------------------
struct Geometry {
    int n_layers, Hq, Hkv, G, d, bs, dtype, es;  // es = element size in bytes
    int out_f32, out_es;                          // output element type / size
    int sink_blocks, local_blocks, budget_blocks, buffer_tokens, reduce, score_mode, select_shared;
    float scale;
};

specpv_status validate_config(const specpv_config* cfg, Geometry* g);
specpv_status validate_kv(const Geometry& g, const specpv_paged_kv* kv);

// Rows of the attention kernels' packed 128-row tiles (floor(128 / G) step tokens each, two tiles per row group).
inline size_t packed_rows(int M_max, int G) {
    const size_t rows = ((size_t)M_max * G + 255) / 256 * 256;
    if (G > 128) return rows;
    const int tok = 128 / G;
    const size_t tiled = (size_t)(M_max + 2 * tok - 1) / (2 * tok) * 256;
    return tiled > rows ? tiled : rows;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- workspace carving --------------------------------------------------------------------
struct WorkspacePlan {
    size_t counter_off, counter_bytes;  // arrival counters of KV ranges shared between CTAs (zero between launches)
    size_t partial_off, partial_bytes;  // split-KV partial results
    size_t staging_off, staging_bytes;  // device copies of host step tensors (specpv_verify_host)
    size_t total;
};
WorkspacePlan plan_workspace(const Geometry& g, int n_layers_per_call, int max_batch, int M_max);

// offsets inside the staging area
struct StagingPlan {
    size_t q, k_new, v_new, mask, out, lse, total;
};
StagingPlan plan_staging(const Geometry& g, int n_layers_per_call, int batch, int M_max);

// ---- dtype helpers ------------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ float to_float(T v);
template <> __device__ __forceinline__ float to_float<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_float(float v);
template <> __device__ __forceinline__ float from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---- launchers implemented in the kernel files --------------------------------------------------
struct AttnArgs {
    Geometry g;
    int layer0, n_layers, batch, M_max, mask_words;
    const void* q;
    const void* k_new;
    const void* v_new;
    const uint64_t* tree_mask;
    const int32_t* q_lens;
    const void* k_pool;
    const void* v_pool;
    const int32_t* block_table;
    const int32_t* seq_lens;
    int max_blocks, n_pages, max_seq_len;
    void* out;
    float* lse;
    void* workspace;
    size_t partial_off, partial_bytes;
    size_t counter_off, counter_bytes;
};

specpv_status launch_attention_simt(const AttnArgs& a, cudaStream_t stream);
specpv_status launch_attention_tc(const AttnArgs& a, cudaStream_t stream);  // bf16
bool attention_tc_supported(const AttnArgs& a);

}  // namespace specpv
