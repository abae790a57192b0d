// Shared device/host helpers of the sdverify kernels.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "sdverify.h"

namespace sdv {

constexpr int kBlock = 64;     // tokens per KV-cache block
constexpr int kD = 128;        // head dimension
constexpr int kMaxT = 64;      // nodes per tree

// first error wins; kernels never trap
__device__ __forceinline__ void set_status(int32_t* status, int code) {
    if (status) atomicCAS(status, 0, code);
}

__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline sd_status cuda_ok(cudaError_t e) { return e == cudaSuccess ? SD_OK : SD_ERR_CUDA; }

// SM count of device `dev` (asked once per device)
int sm_count(int dev);

// Opts a kernel into `bytes` of dynamic shared memory, once per kernel and device (the attribute stays set)
template <typename Kernel>
inline bool allow_dynamic_smem(Kernel* kern, int bytes) {
    struct Done { const void* kern; int dev, bytes; };
    static thread_local Done done[16];                     // (a thread's own, so that no lock is needed)
    static thread_local int next = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    for (const Done& d : done)
        if (d.kern == reinterpret_cast<const void*>(kern) && d.dev == dev && d.bytes >= bytes) return true;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    done[next++ % 16] = Done{reinterpret_cast<const void*>(kern), dev, bytes};
    return true;
}

// Launch that may start while the kernel before it in the stream still runs (programmatic dependent launch):
// the kernel does its set-up and then waits (griddep_wait) for that kernel's completion before it reads or
// writes global memory; every kernel of the library does, so an order of three launches stays an order.
// cluster: CTAs per cluster along x.
template <typename... P, typename... A>
inline sd_status launch_dependent(void (*kern)(P...), dim3 grid, int threads, size_t smem, int cluster, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cuda_ok(cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...));
}

// Start of such a kernel's work on global memory.  The pointers pass through the asm so that no load from
// them, read-only ones included, can be moved in front of the wait.  (The read-only path, __ldg, is for what no kernel
// writes that may still run when this one begins: a caller's inputs, and what the LM-head tiles leave, which let
// nobody begin early.)
template <typename Ptr>
__device__ __forceinline__ void settle(Ptr& p) { asm volatile("" : "+l"(p)); }
__device__ __forceinline__ void settle(sd_batch& bt) {
    settle(bt.block_table); settle(bt.len); settle(bt.n_nodes); settle(bt.parents); settle(bt.anc_mask);
}
template <typename... T>
__device__ __forceinline__ void begin_dependent(T&... p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (settle(p), ...);
}

// Test hooks, read from the environment at every launch (unset in normal use):
//   SDV_TEST_WAIT_CYCLES  bound of the kernels' barrier waits in SM cycles (default: about a second)
//   SDV_TEST_WITHHOLD     1: one role of a kernel withholds its first arrival (draft side: some bytes of every copy),
//                         so that a bounded wait runs out and the launch ends with SD_ERR_TIMEOUT (NaN rows)
//   SDV_TEST_CHUNKS       1 to 8: key chunks per sequence of single-launch attention calls
struct TestKnobs { long long wait_cycles; int withhold; int chunks; };
TestKnobs test_knobs();

// launch-side entry points implemented in the kernel files
sd_status launch_tree_prepare(const sd_batch& bt, int32_t* dev_status, cudaStream_t st);
sd_status launch_accept(const sd_batch& bt, const int32_t* draft, const int32_t* target,
                        int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len,
                        int32_t* dev_status, cudaStream_t st);
sd_status launch_compact(const sd_batch& bt, const sd_kv_layer* layers, int L,
                         const void* const* kt, const void* const* vt,
                         const int32_t* n_acc, const int32_t* path, int32_t* dev_status, cudaStream_t st);
size_t attention_workspace_bytes(const sd_batch& bt);
sd_status launch_attention(const sd_batch& bt, const sd_kv_layer& cache, const void* q,
                           const void* kt, const void* vt, float scale, void* out, float* lse,
                           void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t st);
sd_status launch_attention_layers(const sd_batch& bt, const sd_kv_layer* caches, int L,
                                  const void* const* q, const void* const* kt, const void* const* vt,
                                  float scale, void* const* out, float* const* lse,
                                  int32_t* dev_status, cudaStream_t st);
size_t lmhead_workspace_bytes(int M, int V);
size_t tail_workspace_bytes(int M, int V);
sd_status launch_lmhead(const void* hidden, const void* W, int M, int Hd, int V,
                        int32_t* argmax, float* maxlogit, void* ws, size_t ws_bytes,
                        int32_t* dev_status, cudaStream_t st);

sd_status launch_lmhead_accept_compact(const sd_batch& bt, const void* hidden, const void* W, int Hd, int V,
                                       const int32_t* draft, const sd_kv_layer* layers, int L,
                                       const void* const* kt, const void* const* vt,
                                       int32_t* argmax, float* maxlogit, int32_t* n_acc, int32_t* path,
                                       int32_t* out_tok, int32_t* new_len, void* ws, size_t ws_bytes,
                                       int32_t* dev_status, cudaStream_t st);

sd_status launch_draft_feature_attention(const void* qp, const void* k, const void* v, int S, int L, int Q, int H,
                                         float scale, void* out, cudaStream_t st);
size_t stats_workspace_bytes(int M, int V);
sd_status launch_lmhead_stats(const void* hidden, const void* W, int M, int Hd, int V, float inv_temp,
                              int32_t* argmax, float* maxlogit, float* lse, float* group_stats,
                              void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t st, float* logits = nullptr);
sd_status launch_lmhead_mass(const void* hidden, const void* W, int M, int Hd, int V, float inv_temp,
                             const float* row_lse, float* mass, void* ws, size_t ws_bytes,
                             int32_t* dev_status, cudaStream_t st);
// per-CTA tables the LM-head tiles of a statistics pass leave in the workspace (row stride 512 entries)
struct LmTables { const int32_t* part_key; const int32_t* part_idx; const float* part_ref; const float* part_sum; int n_ctas; };
sd_status launch_lmhead_stats_tiles(const void* hidden, const void* W, int M, int Hd, int V, float inv_temp,
                                    float* lse, float* group_stats, void* ws, size_t ws_bytes,
                                    int32_t* dev_status, cudaStream_t st, LmTables* tables);
size_t sampled_workspace_bytes(int B, int T, int V, int Hd);
sd_status launch_accept_sampled(const sd_batch& bt, const void* hidden, const void* W, int Hd, int V, float inv_temp,
                                const float* lse, const float* group_stats, const int32_t* draft, const float* u,
                                const float* w, int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len,
                                void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t st);

sd_status launch_accept_chain_sampled(const sd_batch& bt, const void* hidden, const void* W, int Hd, int V, float inv_temp,
                                      const float* lse, const float* logits, const int32_t* draft, const float* q_tok,
                                      const float* q_rows, const float* u, const float* w, int32_t* n_acc, int32_t* path,
                                      int32_t* out_tok, int32_t* new_len, void* ws, size_t ws_bytes, int32_t* dev_status,
                                      cudaStream_t st);
bool q_kernels_hold(int V);      // whether a cluster of the kernels for sampled drafts holds a row of V entries
sd_status launch_accept_chain_logits(const sd_batch& bt, int V, float inv_temp, const float* lse, const float* logits,
                                     const int32_t* draft, const float* q_tok, const float* q_rows, const float* u, const float* w,
                                     int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len, int32_t* dev_status,
                                     cudaStream_t st);
sd_status launch_accept_tree_sampled_q(const sd_batch& bt, int V, float inv_temp, const float* lse, const float* logits,
                                       const int32_t* draft, const float* q_rows, const float* u, const float* w,
                                       int32_t* n_acc, int32_t* path, int32_t* out_tok, int32_t* new_len,
                                       int32_t* dev_status, cudaStream_t st);
sd_status launch_lmhead_accept_sampled_compact(const sd_batch& bt, const void* hidden, const void* W, int Hd, int V,
                                               float inv_temp, const int32_t* draft, const float* u, const float* w,
                                               const sd_kv_layer* layers, int L, const void* const* kt, const void* const* vt,
                                               float* lse, float* group_stats, int32_t* n_acc, int32_t* path,
                                               int32_t* out_tok, int32_t* new_len, void* ws, size_t ws_bytes,
                                               int32_t* dev_status, cudaStream_t st);

}  // namespace sdv
