// Internal declarations shared by the CUDA translation units of libgoose.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <initializer_list>

#include "goose.h"

namespace goose {

constexpr int kHeadDim = GOOSE_HEAD_DIM;
constexpr int kMaxB = GOOSE_MAX_B;
constexpr int kMaxK = GOOSE_MAX_K;

// Workspace slot of one split-KV partial.  The mma kernel stores O fp32 [kMaxB][128] (unnormalised), then m[kMaxB],
// l[kMaxB]; the tcgen05 kernel uses the first half of a slot for its fp16 layout (see tree_attn_umma.cu).
constexpr int kPartialFloats = kMaxB * kHeadDim + 2 * kMaxB;

}  // namespace goose

struct goose_ctx {
    int device;
    int num_sms;
    int max_S, max_B, max_H;
    int attn_impl;            // GOOSE_ATTN_*
    // attention workspace
    float* partials;          // [n_slots][kPartialFloats]
    int n_slots;
    int32_t* head_counters;   // [max_S * max_H], zero between launches
    // top-k workspace
    unsigned long long* topk_cand;   // [topk_rows_cap][topk_chunks_cap][kMaxK]
    int32_t* row_counters;    // [topk_rows_cap]
    float* topk_lse_ws;       // [topk_rows_cap][chunks][2]: per-chunk (max, sum) of the log-sum-exp
    int64_t topk_cand_cap;    // elements
    int topk_rows_cap;
    // per-sequence status words
    int32_t* status;          // [max_S]
    int32_t* selftest_word;   // result word of goose_selftest_bounded_wait
    // host staging for goose_verify_step_host
    void* stage;              // device buffer
    size_t stage_bytes;
    void* pin;                // pinned host block: the small input arrays go up, the small results come down, in one copy each
    size_t pin_bytes;
    cudaStream_t side;        // the logits are uploaded here, next to the attention kernels
    cudaStream_t side_down;   // the attention output goes down here while the logits are still going up
    cudaEvent_t ev_fork, ev_logits, ev_attn, ev_out;
    int max_clusters[9];      // clusters of n attention CTAs that the device holds at once, by n
    long long launches;
    void* encode_tiled;       // cuTensorMapEncodeTiled entry point (driver), resolved at create
};

namespace goose {

// Programmatic dependent launch.  Every kernel of the library is launched with the
// programmatic-stream-serialisation attribute and runs  prologue -> pdl_wait() -> pdl_trigger() -> body.
// The prologue takes no result from global memory: it touches none, or only what is final already (inputs of the
// step, ahead of the wait on the step's earlier kernels), or it looks and works out again behind the wait what it saw
// (the tensor-core attention kernel: lengths, counts, rows, its first tile).  pdl_wait() returns once the preceding kernel in the stream has
// completed and its writes are visible; because that kernel passed its own pdl_wait() before it
// triggered, completion is transitive over the whole stream.  The overlap gained is the launch latency
// and the prologue of the next kernel.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Nodes of sequence s: n_nodes[s] when the array is given, else B.  The array is device data: a value outside [0, B]
// reads as 0 (the sequence is skipped like one that has left the batch) and is reported as GOOSE_ST_BAD_NODES.
__host__ __device__ __forceinline__ int nodes_of(const int32_t* __restrict__ n_nodes, int s, int B) {
    if (!n_nodes) return B;
    const int n = n_nodes[s];
    return (n < 0 || n > B) ? 0 : n;
}
__device__ __forceinline__ bool nodes_bad(const int32_t* __restrict__ n_nodes, int s, int B) {
    return n_nodes != nullptr && (n_nodes[s] < 0 || n_nodes[s] > B);
}

// Do a sequence's rows row .. row + ctx + nn - 1 leave the cache?  row and ctx are device data: the sum would wrap for a row
// near 2^63, the differences cannot.
__host__ __device__ __forceinline__ bool rows_outside(int64_t row, int ctx, int nn, int64_t kv_rows) {
    return ctx < 0 || row < 0 || row > kv_rows - nn - ctx;
}

// Bounded mbarrier wait, shared by every kernel that waits on asynchronous copies or tensor-core commits.
// Returns 0 when the barrier phase completed, 1 when `*abort_flag` was raised by another thread of the CTA meanwhile,
// 2 when `limit_cycles` SM cycles passed (the caller raises the flag, records GOOSE_ST_TIMEOUT and unwinds).
__device__ __forceinline__ bool mbar_try_wait_parity(unsigned long long* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ int mbar_wait_bounded(unsigned long long* bar, uint32_t parity, long long limit_cycles,
                                                 volatile int* abort_flag) {
    if (mbar_try_wait_parity(bar, parity)) return 0;
    const long long t0 = clock64();
    for (;;) {
        if (*abort_flag) return 1;
        if (mbar_try_wait_parity(bar, parity)) return 0;
        if (clock64() - t0 > limit_cycles) return 2;
    }
}

// packed fp32 arithmetic: two lanes an instruction
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack_f32x2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, int cluster, size_t smem,
                                      cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    return launch_pdl_cluster(kernel, grid, block, 1, smem, st, args...);
}
#endif

// Where a harvest puts what it finds: logits row r predicts the successors of token row_tok[r], whose row of the dense tables
// [table_rows][k] gets the k ids and their softmax probabilities (a token outside the table: nothing).  Of several rows with one token
// the last one stands.  adj_ids == NULL: no harvest.
struct HarvestTable {
    const int32_t* row_tok;
    int table_rows;
    int32_t* adj_ids;
    float* adj_scores;
};

// Up to this many rows the top-k kernel writes the table, above it a scatter kernel behind it: the scan for later rows with a row's
// token grows with the rows, and in the top-k kernel one warp of an SM has it for all of the SM's rows, one after the other.  Beyond what
// hides beside the stream of a row the whole kernel waits for it.  Harvest, us, scatter kernel -> here (distinct tokens, the longest
// scans):  V = 32000: 600 rows 15.5 -> 14.4, 1500 26.0 -> 25.4, 2048 31.3 -> 31.6, 2500 36.8 -> 39.3, 4000 57 -> 83, 8000 108 -> 470;
// V = 65536: 1000 34.2 -> 31.8, 1500 48.5 -> 46.1, 2048 57.8 -> 57.5, 6000 159 -> 282;  V = 128256: 1500 82.3 -> 82.5, 2048 105.3 ->
// 106.3, 8000 407 -> 642.
constexpr int kTableRows = 1536;

constexpr int kMaxCluster = 8;        // the portable limit

// launchers (each returns a cudaError_t from the launch)
// max_ctas (0: one per SM): the largest grid, beside the attention of a step
// inputs_ready: everything in front of the kernel that precedes this one in the stream is complete when this one can
// start, and that kernel has nothing to do with this one's inputs and outputs (see the kernel)
// table (with row_lse, without n_nodes, at most kTableRows rows): the harvest of every row
// n_nodes (may be NULL) with B: row r = s * B + i exists iff i < n_nodes[s]; other rows are neither read nor written
cudaError_t launch_node_topk(goose_ctx* c, const __nv_bfloat16* logits, int rows, int V, int64_t ldl, int k,
                             int32_t* argmax, int32_t* ids, float* vals, float* row_lse, cudaStream_t st,
                             bool inputs_ready = false, const int32_t* n_nodes = nullptr, int B = 0, int max_ctas = 0,
                             HarvestTable table = {});
// a harvest of more than kTableRows rows: the table, out of the top-k kernel's results
cudaError_t launch_harvest_scatter(goose_ctx* c, const HarvestTable& table, int rows, int k, const int32_t* ids, const float* vals,
                                   const float* row_lse, cudaStream_t st);
cudaError_t launch_accept(goose_ctx* c, const int32_t* draft_tok, const int32_t* parent, const int32_t* n_nodes,
                          const int32_t* argmax, int S, int B, int32_t* path, int32_t* accept_len, int32_t* bonus,
                          cudaStream_t st);
cudaError_t launch_kv_compact(goose_ctx* c, __nv_bfloat16* kc, __nv_bfloat16* vc, const int64_t* row_off,
                              const int32_t* ctx_len, const int32_t* path, const int32_t* accept_len, const int32_t* n_nodes,
                              int S, int B, int H, int64_t kv_rows, int32_t* new_ctx, cudaStream_t st);
cudaError_t launch_accept_compact(goose_ctx* c, __nv_bfloat16* kc, __nv_bfloat16* vc, const int64_t* row_off,
                                  const int32_t* ctx_len, const int32_t* draft_tok, const int32_t* parent,
                                  const int32_t* n_nodes, const int32_t* argmax, int S, int B, int H, int64_t kv_rows, int32_t* path,
                                  int32_t* accept_len, int32_t* bonus, int32_t* new_ctx, cudaStream_t st,
                                  int table_rows = 0, int k = 0, const int32_t* topk_ids = nullptr,
                                  const float* topk_vals = nullptr, const float* row_lse = nullptr,
                                  int32_t* adj_ids = nullptr, float* adj_scores = nullptr,
                                  const struct CombinePlan* merge = nullptr);
cudaError_t launch_tree_attn_mma(goose_ctx* c, const __nv_bfloat16* q, const __nv_bfloat16* kc,
                                 const __nv_bfloat16* vc, int64_t kv_rows, const int64_t* row_off, const int32_t* ctx_len,
                                 const int32_t* parent, const int32_t* n_nodes, int S, int B, int H, int Hkv, float scale,
                                 __nv_bfloat16* out, float* lse, cudaStream_t st);
cudaError_t launch_tree_attn_umma(goose_ctx* c, const __nv_bfloat16* q, const __nv_bfloat16* kc,
                                  const __nv_bfloat16* vc, int64_t kv_rows, const int64_t* row_off,
                                  const int32_t* ctx_len, const int32_t* parent, const int32_t* n_nodes, int S, int B, int H,
                                  int Hkv, float scale, __nv_bfloat16* out, float* lse, cudaStream_t st,
                                  struct CombinePlan* defer_merge = nullptr, int cluster = 0);
// cluster: CTAs a head, 1: the persistent form, 0: the kernel's own choice for a call of its own.
// attn_cluster(): the largest cluster that the device holds, where it pays, else 1;  step: 0 = the attention alone, 1 = in a step, 2 = in a
// step whose top-k is long (more than an item an SM, or with the log-sum-exp).
int attn_heads(int B, int H, int Hkv);                     // heads of the work list of a sequence
bool attn_cluster_fits(const goose_ctx* c, int n, int S, int B, int H, int Hkv, int64_t kv_rows, int step);
int attn_cluster(const goose_ctx* c, int S, int B, int H, int Hkv, int64_t kv_rows, int step);
// a step on device buffers: the attention's cluster size and the top-k's CTAs beside it (0: all SMs, behind the attention)
struct StepSplit { int cluster, topk_ctas; };
StepSplit step_split(const goose_ctx* c, int S, int B, int H, int Hkv, int64_t kv_rows, int V, int k, bool harvest, bool counts);

cudaError_t launch_bounded_wait_selftest(goose_ctx* c, long long limit_cycles, int32_t* result, cudaStream_t st);

// split count of the mma kernel's fixed grid: ctx_len lives on the device, so it depends only on S, H and the SM count
int mma_splits(const goose_ctx* c, int S, int H);

// Called once from goose_create: the kernels are loaded, with their attributes (dynamic shared memory limits), those of a step next to one
// another and the two that no step runs behind them.  Where a kernel's code lies is decided by the order of loading, and three short kernels
// behind one another show it: with the top-k's table form loaded among them steps of 12 us took 0.1 to 0.3 more (32 over 8 heads,
// 16 rows of 32000, 320 keys with the harvest 12.0 -> 12.3; 16 over 2, 32 rows of 128256, 563 keys 11.8 -> 12.0).
inline cudaError_t load_kernels(std::initializer_list<const void*> kernels) {
    cudaFuncAttributes a;
    for (const void* k : kernels)
        if (cudaError_t e = cudaFuncGetAttributes(&a, k)) return e;
    return cudaSuccess;
}
cudaError_t init_mma_kernel();
cudaError_t init_umma_kernel(goose_ctx* c);
cudaError_t init_merge_kernel();
cudaError_t init_topk_kernel();
cudaError_t init_table_kernel();
cudaError_t init_compact_kernel();
cudaError_t init_accept_kernel();
inline cudaError_t init_kernels(goose_ctx* c) {
    cudaError_t e = init_umma_kernel(c);
    for (cudaError_t (*init)() : {init_topk_kernel, init_compact_kernel, init_merge_kernel, init_accept_kernel, init_table_kernel, init_mma_kernel})
        if (e == cudaSuccess) e = init();
    return e;
}

// kernel choice of GOOSE_ATTN_AUTO
int auto_attn_impl(const goose_ctx* c, int S, int B, int H);

}  // namespace goose
