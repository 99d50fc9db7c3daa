// Tree attention on the 5th-generation tensor cores: persistent, warp-specialised kernel
// (tcgen05.mma with TMEM accumulators, TMA loads, mbarrier pipeline).
//
// Work = all (sequence, head, 128-key tile) items in sequence-major order, dealt to the CTAs
// (one per SM) in contiguous ranges, so every SM streams the same number of K/V bytes.  A run of
// items of one head inside a CTA's range is a "segment"; a segment that covers its whole head
// writes the bf16 output directly, any other segment writes a partial (O / l as fp16, running max m and
// running sum l as fp32) to the workspace, and a small second kernel (tree_attn_combine_kernel, spread
// over all SMs) merges the partials of every head that was split.
//
// Roles (192 threads):
//   warp 0, lane 0   TMA producer: Q of the segment, then K and V tiles into a ring of 32 KB stages
//   warp 1, lane 0   MMA issuer:   S = Q K^T into TMEM (double buffered), O += P V into TMEM with P read
//                                  from tensor memory
//   warps 2..5       softmax:      one query row per thread (TMEM lane = row): S from TMEM, ancestor
//                                  mask on the tiles that reach the tree rows, exp2, P (bf16) written back
//                                  over the first 64 columns of the S buffer it came from, lazy rescaling
//                                  of O in TMEM, epilogue (output or partial).
// One sequence that is not too long (kCluster, see attn_cluster): a thread-block cluster takes each head instead, its CTAs
// contiguous tile ranges of it.  No CTA then works on two heads (a second segment costs its softmax, PV and epilogue in
// turn, 2 to 3 us at the end of the slowest CTA), and the cluster merges its head itself, behind its own barrier, instead
// of a kernel behind all of them (boundary 1 us, a cold start on every SM, 2 us, and one more launch).
// All B <= 128 query rows ride in one M = 128 MMA; rows >= B compute on zeros or don't-care data and are
// never written out.  Grouped-query attention (H query heads over Hkv key/value heads, g = H / Hkv) stacks the g
// query heads of a group into the same M tile -- row r = (node r / g, group member r % g) -- so a K/V tile is
// streamed once per group; when B * g > 128 the nodes are cut into M tiles of floor(128 / g) nodes and the K/V of a
// head is streamed once per M tile.  A "head" of the work list below is one (M tile, key/value head) pair.
// The tree part of the mask (Sec. 4 Stage 1: a node attends to the prefix and to its root-to-node ancestors) is a
// per-row 128-bit ancestor set built from parent[].
//
// Every wait in this file is bounded: when a wait runs out of polls the CTA raises an abort flag,
// sets GOOSE_ST_TIMEOUT, drains its own copies in flight (again bounded), frees its TMEM and returns.
#include <cuda.h>
#include <cuda_fp16.h>

#include "goose_internal.cuh"
#include "tree_attn_combine.cuh"

namespace goose {

namespace {

constexpr int kStages = 5;                      // ring of K/V stages (P lives in tensor memory, not here)
constexpr int kStageBytes = kTile * kHeadDim * 2;   // 32 KB: one K or one V tile
constexpr int kHalfBytes = kTile * 128;         // 16 KB: 128 rows x 64 bf16 (one swizzle-atom column)
constexpr int kQBytes = 2 * kHalfBytes;
constexpr int kHeaderBytes = 1024;
constexpr int kUmmaSmem = kHeaderBytes + 1024 /*alignment slack*/ + 2 * kQBytes + kStages * kStageBytes;
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0, kColO = 256;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleThreshold = 8.0f;       // rescale O only when the running max grew by > 2^8
constexpr long long kWaitCycles = 2000000000ll;  // bound of every wait: about one second of SM clock

struct Header {                                  // lives at the start of dynamic shared memory
    unsigned long long kv_full[kStages];
    unsigned long long kv_empty[kStages];
    unsigned long long q_full[2], q_empty[2];    // Q is double buffered: the next segment's Q is prefetched
    unsigned long long s_full[2];
    unsigned long long p_ready, pv_done, o_free;
    unsigned long long group_bar;                // barrier of the 128 softmax threads (bounded, unlike bar.sync)
    uint32_t tmem_base;
    volatile int abort_flag;
    int bad_parent;
    int par[kMaxB];                              // parent[] of the current segment's sequence
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait.  Returns false, and raises the CTA's abort flag, when `limit` SM cycles pass without the barrier
// completing; returns false at once when another role has already aborted.
__device__ __forceinline__ bool mbar_wait_limit(Header* hd, unsigned long long* bar, uint32_t parity, int32_t* status,
                                                long long limit) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
        if (hd->abort_flag) return false;
        if (mbar_try_wait(bar, parity)) return true;
        if (clock64() - t0 > limit) break;
    }
    hd->abort_flag = 1;
    atomicOr(status, GOOSE_ST_TIMEOUT);
    return false;
}
// every wait of the attention kernel: about one second of SM clock
__device__ __forceinline__ bool mbar_wait(Header* hd, unsigned long long* bar, uint32_t parity, int32_t* status) {
    return mbar_wait_limit(hd, bar, parity, status, kWaitCycles);
}
// Bounded wait used only while draining after an abort (ignores the abort flag).
__device__ __forceinline__ void mbar_drain(unsigned long long* bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity) && clock64() - t0 < kWaitCycles) {}
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, unsigned long long* bar,
                                            int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_3d_hint(void* dst, const CUtensorMap* map, unsigned long long* bar,
                                                 int c0, int c1, int c2, unsigned long long policy) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
                 "[%0], [%1, {%3, %4, %5}], [%2], %6;"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}
// brings a box of a tensor map into L2: a hint; nothing reaches the SM, and a box outside the tensor touches nothing
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap* map, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];" ::"l"(map), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// a load that may run beside the kernel that writes the word (it returns the old or the new value)
__device__ __forceinline__ int32_t load_early(const int32_t* p) {
    int32_t v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int64_t load_early(const int64_t* p) {
    int64_t v;
    asm volatile("ld.relaxed.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long l2_policy_evict_first() {
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle (addresses and offsets in bytes): the half that holds the address (in a
// cluster the bits above say which CTA's: cut off), to which an offset / 16 may be added as long as the sum stays in shared
// memory, and the other half, the same for all.  One descriptor a tile and additions instead of sixteen built from scratch by
// the issuing thread, and tile counts and stages carried along instead of worked out tile by tile (with 64-bit list positions
// and divisions by five), stood between a tile's arrival and its scores: attention call 512 keys 8.5 -> 8.1, 1531 11.4 -> 11.0,
// 2k 12.7 -> 12.4, 8k 28.0 -> 27.4 (32 heads), 32 over 8 heads 3k 12.2 -> 11.9, 2 x 32 over 8 16.7 -> 16.4 us, with the
// multiplication of cluster_start(), to which the clusters owe most of it.
__device__ __forceinline__ uint32_t smem_desc_lo(uint32_t addr, uint32_t lbo) { return ((addr >> 4) & 0x3FFF) | ((lbo >> 4) << 16); }
__device__ __forceinline__ uint64_t smem_desc(uint32_t lo) {
    constexpr uint32_t hi = (1024u >> 4) /*SBO: the next eight rows*/ | (1u << 14) /*descriptor version*/ | (2u << 29) /*SWIZZLE_128B*/;
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}
// instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = 128, A K-major, B K-major or MN-major
__host__ __device__ constexpr uint32_t instr_desc(bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// same, with the A operand (M x 16 bf16, two per 32-bit column, lane = row) read from tensor memory
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// the cluster's barrier: orders the partials written by its CTAs before the reads behind it
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
#define TMEM_LD32(taddr, v, off)                                                                                      \
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "                                                            \
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"                                          \
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"                           \
                 : "=r"(v[off + 0]), "=r"(v[off + 1]), "=r"(v[off + 2]), "=r"(v[off + 3]), "=r"(v[off + 4]),          \
                   "=r"(v[off + 5]), "=r"(v[off + 6]), "=r"(v[off + 7]), "=r"(v[off + 8]), "=r"(v[off + 9]),          \
                   "=r"(v[off + 10]), "=r"(v[off + 11]), "=r"(v[off + 12]), "=r"(v[off + 13]), "=r"(v[off + 14]),     \
                   "=r"(v[off + 15]), "=r"(v[off + 16]), "=r"(v[off + 17]), "=r"(v[off + 18]), "=r"(v[off + 19]),     \
                   "=r"(v[off + 20]), "=r"(v[off + 21]), "=r"(v[off + 22]), "=r"(v[off + 23]), "=r"(v[off + 24]),     \
                   "=r"(v[off + 25]), "=r"(v[off + 26]), "=r"(v[off + 27]), "=r"(v[off + 28]), "=r"(v[off + 29]),     \
                   "=r"(v[off + 30]), "=r"(v[off + 31])                                                               \
                 : "r"(taddr))
#define TMEM_ST32(taddr, v, off)                                                                                      \
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "                                                     \
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"                                          \
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};"                                  \
                 ::"r"(v[off + 0]), "r"(v[off + 1]), "r"(v[off + 2]), "r"(v[off + 3]), "r"(v[off + 4]),               \
                   "r"(v[off + 5]), "r"(v[off + 6]), "r"(v[off + 7]), "r"(v[off + 8]), "r"(v[off + 9]),               \
                   "r"(v[off + 10]), "r"(v[off + 11]), "r"(v[off + 12]), "r"(v[off + 13]), "r"(v[off + 14]),          \
                   "r"(v[off + 15]), "r"(v[off + 16]), "r"(v[off + 17]), "r"(v[off + 18]), "r"(v[off + 19]),          \
                   "r"(v[off + 20]), "r"(v[off + 21]), "r"(v[off + 22]), "r"(v[off + 23]), "r"(v[off + 24]),          \
                   "r"(v[off + 25]), "r"(v[off + 26]), "r"(v[off + 27]), "r"(v[off + 28]), "r"(v[off + 29]),          \
                   "r"(v[off + 30]), "r"(v[off + 31]), "r"(taddr) : "memory")

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// barrier of the 128 softmax threads; `n` counts its uses (every thread calls it the same number of times)
__device__ __forceinline__ bool group_sync(Header* hd, uint32_t& n, int32_t* status) {
    mbar_arrive(&hd->group_bar);
    bool ok = mbar_wait(hd, &hd->group_bar, n & 1, status);
    ++n;
    return ok;
}

// ---------------------------------------------------------------- the kernel
// kGrouped = false is multi-head attention: one query head per key/value head and one M tile per sequence are
// compile-time facts there (the per-row index arithmetic folds away); kGrouped = true takes them from the arguments.
// kCounts = false is the instantiation for n_nodes == NULL: the counts fold away at compile time
template <bool kGrouped, bool kCounts, bool kCluster>
__global__ void __launch_bounds__(kThreads, 1)
tree_attn_umma_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                      const __grid_constant__ CUtensorMap tmap_v, const int64_t* __restrict__ row_off,
                      const int32_t* __restrict__ ctx_len, const int32_t* __restrict__ parent,
                      const int32_t* __restrict__ n_nodes,
                      int S, int B, int H, int Hkv_arg, int g_arg, int nb_arg, uint32_t G_magic, int cluster, int64_t kv_rows,
                      float scale_log2,
                      float* __restrict__ partials,
                      int32_t* __restrict__ status,
                      __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
    if (!kCounts) n_nodes = nullptr;

    const int Hkv = kGrouped ? Hkv_arg : H, g = kGrouped ? g_arg : 1, nb = kGrouped ? nb_arg : B;
    extern __shared__ unsigned char smem_raw[];
    Header* hd = reinterpret_cast<Header*>(smem_raw);
    unsigned char* buf = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + kHeaderBytes + 1023) & ~(uintptr_t)1023);
    unsigned char* q_smem = buf;
    unsigned char* kv_smem = buf + 2 * kQBytes;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // ---- set-up
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(&hd->kv_full[i], 1); mbar_init(&hd->kv_empty[i], 1); }
        mbar_init(&hd->q_full[0], 1); mbar_init(&hd->q_full[1], 1);
        mbar_init(&hd->q_empty[0], 1); mbar_init(&hd->q_empty[1], 1);
        mbar_init(&hd->s_full[0], 1); mbar_init(&hd->s_full[1], 1);
        mbar_init(&hd->p_ready, 128); mbar_init(&hd->pv_done, 1); mbar_init(&hd->o_free, 128);
        mbar_init(&hd->group_bar, 128);
        hd->abort_flag = 0; hd->bad_parent = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {                                   // TMEM: the whole 512 columns (one CTA per SM)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&hd->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) { prefetch_tmap(&tmap_q); prefetch_tmap(&tmap_k); prefetch_tmap(&tmap_v); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = hd->tmem_base;
    // L2 prefetch hints for the small index arrays (a hint reads no data, so it may precede the wait)
    if (threadIdx.x == 32) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(ctx_len));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(row_off));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(parent));
    }
    Work wk;
    // g query heads per key/value head, nb nodes per M tile (nb * g <= 128), n_mt M tiles per sequence
    const int n_mt = kGrouped ? (B + nb - 1) / nb : 1;
    wk.ctx_len = ctx_len; wk.n_nodes = n_nodes; wk.S = S; wk.H = n_mt * Hkv; wk.B = B; wk.G = gridDim.x; wk.G_magic = G_magic;
    wk.kv_rows = (int)kv_rows;                          // (the entry points take no more than 2^31 - 1)
    // cluster mode: this CTA is number `rank` of the `cluster` CTAs that share head `head` of the one sequence
    const int head = kCluster ? (int)__umulhi(blockIdx.x, G_magic) : 0, rank = kCluster ? blockIdx.x - head * cluster : 0;
    int T_all = 0;                                      // tiles of that sequence
    auto rank_start = [&](int r) { return cluster_start(T_all, r, cluster, G_magic); };
    // this CTA's items, found by a whole warp (lane = sequence, `tiles` its tiles); a list of more than 32 sequences is read again
    long long w_begin = 0, w_end = 0;
    Cursor cu;
    auto locate = [&](int tiles, int lane) {
        if (kCluster) {
            T_all = __shfl_sync(0xFFFFFFFFu, tiles, 0);
            w_begin = (long long)head * T_all + rank_start(rank); w_end = (long long)head * T_all + rank_start(rank + 1);
            cu.w = w_begin; cu.s = 0; cu.h = head; cu.t = rank_start(rank); cu.T = T_all;
        } else {
            w_begin = wk.cta_start(blockIdx.x); w_end = wk.cta_start(blockIdx.x + 1);
            if (w_begin < w_end) {
                cu.seek_warp(wk, w_begin, lane, tiles);
                if (!cu.any(w_end)) w_end = w_begin;    // idle items alone: no work, and no tile to look at ahead of the wait
            }
        }
    };
    // The CTA is up 0.7 to 1 us before the kernel in front has ended, and the first load of K after that used to take 1.8 us.
    // One warp brings the CTA's first tile into L2 meanwhile: where it lies is worked out from lengths that the kernel in front
    // may still be writing, so all of it is a hint, worked out again below.  Attention call without -> with, us: 32 heads 512 keys
    // 9.2 -> 8.6, 1531 12.4 -> 11.6, 2k 13.6 -> 12.9, 8k 29.2 -> 28.3; 52 heads 8k 43.7 -> 42.0; 4 x 32 over 8, 4k to 16k 41.1 -> 39.8.
    // That is behind a kernel of this library, which lets its dependents in as soon as its own wait is over.  Behind one that does
    // not, the CTA comes up when the lengths are final and there is little time to gain (a small element-wise kernel, then the call;
    // both, without -> with the look and the places below): 512 10.9 to 11.4 -> 10.9, 1531 14.1 to 14.6 -> 13.9 to 14.7.
    // (Two tiles and more, or by CTAs on idle SMs all of the next call's tiles: slower, 2k 14.1 and more.  The copies in flight
    // are then so many that HBM delivers less.)
    // Multi-head: all warps work their place out here, and where the lengths behind the wait are the same (they are, unless the kernel
    // in front writes them) it stands: step of 32 heads at 2k 17.0 -> 16.7, 40 heads 4k 25.3 -> 24.9, 52 heads 8k 45.5 -> 45.2, 8 ragged
    // sequences 85.5 -> 84.5.  Grouped-query heads look again: with the place kept, call of 4 x 32 over 8 35.4 -> 35.7, 2 x 32 over 8
    // 17.0 -> 17.6, one sequence in clusters 12.10 -> 12.01 and its cycle 20.6 -> 20.7.
    int early_ctx = 0, early_nn = 0;
    bool placed = false;
    if (S <= 32 && (!kGrouped || warp == 2)) {
        const bool mine = lane < S;
        early_nn = !mine ? 0 : kCounts ? load_early(n_nodes + lane) : B;
        early_ctx = mine ? load_early(ctx_len + lane) : 0;
        const int64_t row0 = warp == 2 && mine ? load_early(row_off + lane) : 0;
        const int tiles = early_nn > 0 && early_nn <= B ? wk.tiles_of(early_ctx, early_nn) : 0;
        wk.init_lanes(tiles, tiles > 0);
        placed = kCluster || wk.small;                  // (a longer list is walked through lengths in memory: not yet)
        if (placed) locate(tiles, lane);
        if (warp == 2 && placed && w_begin < w_end) {
            const int64_t first = __shfl_sync(0xFFFFFFFFu, row0, cu.s), row = min(first, kv_rows) + (int64_t)cu.t * kTile;
            if (lane < 4 && first >= 0 && row < kv_rows)
                tma_prefetch_3d(lane & 2 ? &tmap_v : &tmap_k, (lane & 1) * 64, kGrouped ? cu.h % Hkv : cu.h, (int)row);
        }
    }
    // everything above only looked: now wait for the preceding kernel, then let the next
    // one (the combine kernel) get resident early -- it waits for this grid before reading the partials
    pdl_wait();
    pdl_trigger();
    if (n_nodes && blockIdx.x == 0 && threadIdx.x == 33)   // an idle lane reports node counts outside [0, B] (read as 0)
        for (int s = 0; s < S; ++s)
            if (nodes_bad(n_nodes, s, B)) atomicOr(&status[s], GOOSE_ST_BAD_NODES);
    // where this CTA starts, found by every warp for itself with all lanes; the lengths and the rows of up to 32 sequences
    // come in one round of loads (lane = sequence).  The first load of K waits for nothing else.
    const int64_t my_row = lane < S ? row_off[lane] : 0;
    if (kGrouped) {
        locate(wk.init_warp(lane), lane);
    } else {
        const bool same = placed && (lane >= S || (ctx_len[lane] == early_ctx && (!kCounts || n_nodes[lane] == early_nn)));
        if (!__all_sync(0xFFFFFFFFu, same)) locate(wk.init_warp(lane), lane);
    }
    const int first_s = w_begin < w_end ? cu.s : 0;
    const int64_t first_row = __shfl_sync(0xFFFFFFFFu, my_row, first_s & 31);
    auto row_of = [&](int s) -> int64_t { return s == first_s && s < 32 ? first_row : row_off[s]; };


    if (w_begin < w_end) {
        if (warp == 0) {
            // =========================================================== TMA producer
            if (lane == 0) {
                // K and V are read exactly once: mark them evict-first so that the split-KV partials
                // (written and re-read within this launch) stay resident in L2
                const unsigned long long pol_stream = l2_policy_evict_first();
                uint32_t ring = 0, st = 0, phase = 0, seg = 0;   // copies issued; the stage of the next and its phase
                bool ok = true;
                while (ok && cu.w < w_end) {
                    const int64_t row0 = row_of(cu.s);
                    // Q of this segment
                    const uint32_t qb = seg & 1;           // seg = index of this segment
                    ok = mbar_wait(hd, &hd->q_empty[qb], ((seg >> 1) & 1) ^ 1, status);
                    if (!ok) break;
                    // box = nb nodes x g heads x 64 dims: lands as rows r = node * g + member (rows past the
                    // sequence's last node hold the next sequence's queries or the zero fill: never written out)
                    const int mt = kGrouped ? cu.h / Hkv : 0, hk = cu.h - mt * Hkv;
                    mbar_expect_tx(&hd->q_full[qb], (uint32_t)(nb * g) * 256u);
                    tma_load_4d(q_smem + qb * kQBytes, &tmap_q, &hd->q_full[qb], 0, 0, hk, cu.s * B + mt * nb);
                    tma_load_4d(q_smem + qb * kQBytes + kHalfBytes, &tmap_q, &hd->q_full[qb], 64, 0, hk, cu.s * B + mt * nb);
                    ++seg;                                 // segments whose Q load has been issued
                    const int n = cu.run(w_end);
                    int krow = (int)(row0 + (int64_t)cu.t * kTile);
                    for (int i = 0; i < n && ok; ++i, krow += kTile) {
                        for (int kv = 0; kv < 2 && ok; ++kv) {
                            ok = mbar_wait(hd, &hd->kv_empty[st], phase ^ 1, status);
                            if (!ok) break;
                            unsigned char* dst = kv_smem + st * kStageBytes;
                            mbar_expect_tx(&hd->kv_full[st], kStageBytes);
                            const CUtensorMap* mp = kv ? &tmap_v : &tmap_k;
                            tma_load_3d_hint(dst, mp, &hd->kv_full[st], 0, hk, krow, pol_stream);
                            tma_load_3d_hint(dst + kHalfBytes, mp, &hd->kv_full[st], 64, hk, krow, pol_stream);
                            ++ring;
                            if (++st == kStages) { st = 0; phase ^= 1; }
                        }
                    }
                    cu.skip(wk, n);
                }
                if (!ok) {
                    // aborted: drain this thread's copies still in flight (bounded) before the CTA exits
                    uint32_t first = ring > kStages ? ring - kStages : 0;
                    for (uint32_t r = first; r < ring; ++r) mbar_drain(&hd->kv_full[r % kStages], (r / kStages) & 1);
                    if (seg > 0) mbar_drain(&hd->q_full[(seg - 1) & 1], ((seg - 1) >> 1) & 1);
                    if (seg > 1) mbar_drain(&hd->q_full[(seg - 2) & 1], ((seg - 2) >> 1) & 1);
                }
            }
        } else if (warp == 1) {
            // =========================================================== MMA issuer
            if (lane == 0) {
                uint32_t jg = 0, seg = 0;                  // CTA-global tile and segment counters
                bool ok = true;
                const uint32_t q_base = smem_u32(q_smem), kv_addr = smem_u32(kv_smem);
                constexpr uint32_t idesc_qk = instr_desc(false), idesc_pv = instr_desc(true);

                // stage and phase of the next K tile and of the next V tile: every second stage of the ring
                uint32_t k_st = 0, k_phase = 0, v_st = 1, v_phase = 0;
                auto next_stage = [](uint32_t& st, uint32_t& phase) {
                    st += 2;
                    if (st >= kStages) { st -= kStages; phase ^= 1; }
                };
                auto issue_pv = [&](uint32_t j, bool first_of_segment) -> bool {
                    // tile j's P (bf16) has replaced S(j) in the first 64 columns of its S buffer
                    if (!mbar_wait(hd, &hd->p_ready, j & 1, status)) return false;
                    if (!mbar_wait(hd, &hd->kv_full[v_st], v_phase, status)) return false;
                    if (first_of_segment && seg > 0)       // the previous segment's O must have left TMEM
                        if (!mbar_wait(hd, &hd->o_free, (seg - 1) & 1, status)) return false;
                    tc_fence_after();
                    const uint32_t v_lo = smem_desc_lo(kv_addr + v_st * kStageBytes, kHalfBytes);   // MN-major: LBO = next 64 d
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {       // 16 keys per instruction
                        umma_f16_ts(tmem + kColO, tmem + kColS + (j & 1) * 128 + kk * 8, smem_desc(v_lo + kk * (2048 >> 4)), idesc_pv,
                                    (!first_of_segment || kk > 0) ? 1u : 0u);
                    }
                    umma_commit(&hd->kv_empty[v_st]);
                    umma_commit(&hd->pv_done);
                    next_stage(v_st, v_phase);
                    return true;
                };

                while (ok && cu.w < w_end) {
                    ok = mbar_wait(hd, &hd->q_full[seg & 1], (seg >> 1) & 1, status);
                    if (!ok) break;
                    const uint32_t q_lo = smem_desc_lo(q_base + (seg & 1) * kQBytes, 16);
                    const int n = cu.run(w_end);
                    const uint32_t j_first = jg;
                    for (int i = 0; i < n && ok; ++i) {
                        ok = mbar_wait(hd, &hd->kv_full[k_st], k_phase, status);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t k_lo = smem_desc_lo(kv_addr + k_st * kStageBytes, 16);
                        const uint32_t d_tmem = tmem + kColS + (jg & 1) * 128;
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk) {   // 16 of the 128 head dims per instruction
                            const uint32_t off = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
                            umma_f16(d_tmem, smem_desc(q_lo + off), smem_desc(k_lo + off), idesc_qk, kk > 0 ? 1u : 0u);
                        }
                        umma_commit(&hd->s_full[jg & 1]);
                        umma_commit(&hd->kv_empty[k_st]);
                        next_stage(k_st, k_phase);
                        if (jg > j_first) ok = issue_pv(jg - 1, jg - 1 == j_first);
                        ++jg;
                    }
                    if (!ok) break;
                    cu.skip(wk, n);
                    umma_commit(&hd->q_empty[seg & 1]);    // every QK^T of the segment has been issued
                    ok = issue_pv(jg - 1, jg - 1 == j_first);
                    ++seg;
                }
            }
        } else {
            // =========================================================== softmax / epilogue (128 threads)
            const int row = 32 * (warp & 3) + lane;        // TMEM lane == query row
            const uint32_t lane_sel = (uint32_t)(32 * (warp & 3)) << 16;
            const int i_local = kGrouped ? row / g : row;  // row = (node of the M tile, head of the group)
            const int member = row - i_local * g;
            const int sm_tid = threadIdx.x - 64;           // 0..127
            uint32_t jg = 0, seg = 0, gsync = 0;
            bool ok = true;
            uint32_t v[128];
            int cur_s = -1, cur_mt = -1;
            bool bad = false, anc_built = false;
            uint32_t anc[4] = {0, 0, 0, 0};
            // Rows of the M tile that no query fills: zeros instead of what shared memory held.  No result depends on them (and so
            // nothing waits for these stores), but a long stream is held back by the power that the card may draw, and products of
            // zeros draw less: steps under continuous load, 16 x 32 heads 1k to 16k with 64 rows 445 -> 426 us, 7 ragged sequences of
            // 32 heads with at most 60 rows 92.4 -> 90.0; 40 heads 4k with 80 rows even.  By the softmax threads, which wait
            // for the first scores here; in the set-up, ahead of the dependency wait, it cost short calls 0.3 to 0.4 us.
            if (!kCluster) {
                for (int off = nb * g * 128 + sm_tid * 16; off < kHalfBytes; off += 128 * 16) {
#pragma unroll
                    for (int half = 0; half < 4; ++half) *reinterpret_cast<uint4*>(q_smem + half * kHalfBytes + off) = make_uint4(0, 0, 0, 0);
                }
            }

            while (ok && cu.w < w_end) {
                const int s0 = cu.s, h0 = cu.h, T = cu.T;
                const int mt = kGrouped ? h0 / Hkv : 0, hk = h0 - mt * Hkv;
                const int node = mt * nb + i_local;        // tree node of this thread's row
                const int nn = nodes_of(n_nodes, s0, B);   // nodes this sequence's tree really has (> 0: it has items)
                const bool row_valid = i_local < nb && node < nn;
                const bool warp_has_rows = 32 * (warp & 3) < min(nb, nn - mt * nb) * g;
                const int ctx = wk.prefix(ctx_len[s0]);
                const int n_keys = ctx + nn;               // rows behind may hold anything: masked, and zeroed in V
                const int32_t* par = parent + (size_t)s0 * B;
                const int t_first = cu.t;
                // new sequence: validate parent[] (all 128 threads reach the same verdict) and rebuild
                // this row's ancestor set; consecutive segments of one sequence reuse both
                const bool new_seq = s0 != cur_s;
                if (new_seq) {
                    cur_s = s0;
                    if (row < nn) {                        // thread r stages parent[r] (independent of the row stacking)
                        int p = par[row];
                        hd->par[row] = p;
                        if ((row == 0) ? (p != -1) : (p < 0 || p >= row)) hd->bad_parent = 1;
                    }
                    // the sequence's rows must lie inside the cache (TMA would only read zeros outside, but the
                    // result would be meaningless): treated like an invalid tree, with its own status bit
                    const bool bad_rows = rows_outside(row_of(s0), ctx_len[s0], nn, kv_rows);
                    if (bad_rows && sm_tid == 0) { hd->bad_parent = 1; atomicOr(&status[s0], GOOSE_ST_BAD_ROWS); }
                    ok = group_sync(hd, gsync, status);
                    bad = hd->bad_parent != 0;
                    ok = ok && group_sync(hd, gsync, status);
                    if (!ok) break;
                    if (sm_tid == 0 && bad) { hd->bad_parent = 0; if (!bad_rows) atomicOr(&status[s0], GOOSE_ST_BAD_PARENT); }
                }
                if (new_seq || mt != cur_mt) {
                    cur_mt = mt;
                    anc_built = false;
                }
                // the ancestor set of this thread's row, for segments that reach the tree rows (hd->par[] still holds this
                // sequence's parents)
                const int t_end = t_first + cu.run(w_end);
                if (!anc_built && t_end * kTile > ctx) {
                    anc_built = true;
                    anc[0] = anc[1] = anc[2] = anc[3] = 0;
                    if (row_valid) {
                        if (bad) {
                            const uint32_t bit = 1u << (node & 31);
                            const int wsel = node >> 5;
                            anc[0] = (wsel == 0) ? bit : 0; anc[1] = (wsel == 1) ? bit : 0;
                            anc[2] = (wsel == 2) ? bit : 0; anc[3] = (wsel == 3) ? bit : 0;
                        } else {
                            int vtx = node;
                            for (int step = 0; step < B && vtx >= 0; ++step) {
                                uint32_t bit = 1u << (vtx & 31);
                                int wsel = vtx >> 5;
                                anc[0] |= (wsel == 0) ? bit : 0; anc[1] |= (wsel == 1) ? bit : 0;
                                anc[2] |= (wsel == 2) ? bit : 0; anc[3] |= (wsel == 3) ? bit : 0;
                                vtx = hd->par[vtx];
                            }
                        }
                    }
                }
                float m_run = -INFINITY, l_run = 0.f;

                for (int t = t_first; t < t_end; ++t) {
                    const bool first = (t == t_first);
                    ok = mbar_wait(hd, &hd->s_full[jg & 1], (jg >> 1) & 1, status);
                    if (!ok) break;
                    tc_fence_after();
                    // The maximum stands in front of the exponentials.  Taken beside them, relative to the older maximum and with
                    // a second pass over a tile whose maximum grew by more than the threshold, the tile's registers did not
                    // fit (20 to 112 bytes of spill loads in every instantiation) and such a tile cost twice.  Attention call
                    // beside -> in front, us: 32 heads 4k 20.4 -> 18.9, 52 heads 8k 44.1 -> 43.5, 8 x 32 heads 16k 336 -> 328,
                    // 32 over 8 heads 16k 30.0 -> 28.6; scores that rise by 2^9 a tile, 4 x 32 heads 2k to 8k 66.9 -> 48.9.
                    if (warp_has_rows) {
                        const uint32_t s_addr = tmem + kColS + (jg & 1) * 128 + lane_sel;
                        TMEM_LD32(s_addr, v, 0); TMEM_LD32(s_addr + 32, v, 32);
                        TMEM_LD32(s_addr + 64, v, 64); TMEM_LD32(s_addr + 96, v, 96);
                        tmem_wait_ld();
                        const int key0 = t * kTile;
                        if (key0 + kTile > ctx) {          // this tile reaches the tree rows (or the ragged end)
                            // visibility of the tile's 128 keys as one 128-bit mask: the prefix keys
                            // (c < ctx - key0) and the ancestor set shifted to where the tree rows start
                            const int pc = ctx - key0;     // tile column of tree node 0 (may be < 0 or >= 128)
                            const unsigned __int128 a128 =
                                ((unsigned __int128)(((unsigned long long)anc[3] << 32) | anc[2]) << 64) |
                                (unsigned __int128)(((unsigned long long)anc[1] << 32) | anc[0]);
                            unsigned __int128 vm;
                            if (pc >= 128) vm = ~(unsigned __int128)0;
                            else if (pc > 0) vm = (((unsigned __int128)1 << pc) - 1) | (a128 << pc);
                            else if (pc > -128) vm = a128 >> (-pc);
                            else vm = 0;
                            const uint32_t vw[4] = {(uint32_t)vm, (uint32_t)(vm >> 32), (uint32_t)(vm >> 64), (uint32_t)(vm >> 96)};
#pragma unroll
                            for (int c = 0; c < 128; ++c)
                                v[c] = ((vw[c >> 5] >> (c & 31)) & 1u) ? v[c] : 0xFF800000u;   // -inf
                        }
                        // one warp per scheduler: nothing hides a serial chain, so the row maximum (and the row sum below)
                        // run as four independent chains
                        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int c = 0; c < 128; c += 8)
#pragma unroll
                            for (int e = 0; e < 4; ++e) mx4[e] = max3(mx4[e], __uint_as_float(v[c + 2 * e]), __uint_as_float(v[c + 2 * e + 1]));
                        const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * scale_log2;   // scale > 0
                        const float m_new = fmaxf(m_run, mx);
                        // lazy rescaling: keep the stale maximum unless it grew by more than the threshold (in a row that
                        // exists: the others hold whatever shared memory held, and results may not depend on that)
                        if (__any_sync(0xFFFFFFFFu, first || (row_valid && m_new > m_run + kRescaleThreshold))) {
                            const float alpha = (m_run == -INFINITY) ? 0.f : ex2(m_run - m_new);
                            if (!first) {
                                // O holds tiles < t of this segment: wait for PV(t-1), then scale the row
                                ok = mbar_wait(hd, &hd->pv_done, (jg - 1) & 1, status);
                                if (ok) {
                                    tc_fence_after();
                                    uint32_t o[32];
                                    const uint32_t o_addr = tmem + kColO + lane_sel;
#pragma unroll
                                    for (int cc = 0; cc < 4; ++cc) {
                                        TMEM_LD32(o_addr + cc * 32, o, 0);
                                        tmem_wait_ld();
#pragma unroll
                                        for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
                                        TMEM_ST32(o_addr + cc * 32, o, 0);
                                    }
                                    tmem_wait_st();
                                }
                            }
                            l_run *= alpha;
                            m_run = m_new;
                        }
                        const float neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
                        const unsigned long long scale2 = pack_f32x2(scale_log2, scale_log2), neg2 = pack_f32x2(neg_m, neg_m);
                        unsigned long long ls2[2] = {0, 0};
#pragma unroll
                        for (int e = 0; e < 64; ++e) {
                            const float2 x2 = unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), scale2, neg2));
                            const float p0 = ex2(x2.x), p1 = ex2(x2.y);
                            ls2[e & 1] = add_f32x2(ls2[e & 1], pack_f32x2(p0, p1));
                            v[e] = pack_bf16x2(p0, p1);
                        }
                        const float2 l2 = unpack_f32x2(add_f32x2(ls2[0], ls2[1]));
                        l_run += l2.x + l2.y;
                        // P (bf16 pairs) overwrites the first 64 columns of this tile's S buffer: this thread has its whole
                        // S row in registers, and QK^T of tile jg+2 is ordered after PV(jg) in the MMA pipe
                        const uint32_t p_taddr = tmem + kColS + (jg & 1) * 128 + lane_sel;
                        TMEM_ST32(p_taddr, v, 0);
                        TMEM_ST32(p_taddr + 32, v, 32);
                        tmem_wait_st();
                    }
                    // observe every phase of pv_done in order (a parity wait must never lag two phases behind its
                    // barrier); by now PV(jg-1) has normally completed, so this does not stall
                    if (ok && jg > 0) ok = mbar_wait(hd, &hd->pv_done, (jg - 1) & 1, status);
                    if (!ok) break;
                    // ragged end: V rows past the sequence's last key may hold anything -> zero them
                    if ((t + 1) * kTile > n_keys) {
                        const uint32_t ring = 2 * jg + 1, st = ring % kStages;
                        ok = mbar_wait(hd, &hd->kv_full[st], (ring / kStages) & 1, status);
                        if (!ok) break;
                        // rows n_keys - t * 128 .. 127 are one contiguous piece of each half (the swizzle stays inside a
                        // row): consecutive threads clear consecutive 16-byte words.  (A row per thread had all lanes of
                        // a store on the same four banks: 0.5 to 0.9 us on the last tile of every head.)
                        const int first_off = max(n_keys - t * kTile, 0) * 128;
                        for (int off = first_off + sm_tid * 16; off < kHalfBytes; off += 128 * 16) {
                            *reinterpret_cast<uint4*>(kv_smem + st * kStageBytes + off) = make_uint4(0, 0, 0, 0);
                            *reinterpret_cast<uint4*>(kv_smem + st * kStageBytes + kHalfBytes + off) = make_uint4(0, 0, 0, 0);
                        }
                        fence_proxy_async();               // generic-proxy writes -> visible to the tensor core
                    }
                    tc_fence_before();
                    mbar_arrive(&hd->p_ready);
                    ++jg;
                }
                if (!ok) break;
                cu.skip(wk, t_end - t_first);

                // ---------------- segment epilogue: O of tiles [t_first, t_end) is complete after PV(jg-1)
                ok = mbar_wait(hd, &hd->pv_done, (jg - 1) & 1, status);
                if (!ok) break;
                tc_fence_after();
                const bool whole_head = t_first == 0 && t_end == T;
                if (warp_has_rows) {
                    const uint32_t o_addr = tmem + kColO + lane_sel;
                    TMEM_LD32(o_addr, v, 0); TMEM_LD32(o_addr + 32, v, 32);
                    TMEM_LD32(o_addr + 64, v, 64); TMEM_LD32(o_addr + 96, v, 96);
                    tmem_wait_ld();
                }
                tc_fence_before();
                mbar_arrive(&hd->o_free);                  // TMEM O may be overwritten by the next segment

                const int hq = hk * g + member;            // query head of this row
                if (whole_head) {
                    if (row_valid) {
                        const float inv = bad ? 0.f : 1.f / l_run;
                        uint4* dst = reinterpret_cast<uint4*>(out + (((size_t)s0 * B + node) * H + hq) * kHeadDim);
#pragma unroll
                        for (int ch = 0; ch < 16; ++ch) {
                            uint32_t pk[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                pk[e] = bad ? 0u : pack_bf16x2(__uint_as_float(v[ch * 8 + 2 * e]) * inv,
                                                               __uint_as_float(v[ch * 8 + 2 * e + 1]) * inv);
                            dst[ch] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                        if (lse) lse[((size_t)s0 * B + node) * H + hq] = bad ? 0.f : (m_run + log2f(l_run)) * kLn2;
                    }
                } else {
                    // partial -> workspace slot of this CTA (combined by tree_attn_combine_kernel): O/l in fp16
                    // (relative error 2^-11, far below the bf16 rounding of the final output), m and l in fp32
                    const int slot = kCluster ? blockIdx.x : 2 * blockIdx.x + (t_first == 0 ? 1 : 0);
                    float* part = partials + (size_t)slot * kUmmaPartFloats;
                    if (row_valid) {
                        // invalid parent[]: a neutral partial (O = 0; the head's first part carries weight 1)
                        // makes the combine kernel produce the defined zero output without re-validating
                        const float inv = (bad || l_run == 0.f) ? 0.f : 1.f / l_run;
                        uint4* dst = reinterpret_cast<uint4*>(part) + row;
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            uint32_t hw[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                __half2 h2 = __floats2half2_rn(__uint_as_float(v[8 * c + 2 * e]) * inv,
                                                               __uint_as_float(v[8 * c + 2 * e + 1]) * inv);
                                hw[e] = *reinterpret_cast<uint32_t*>(&h2);
                            }
                            dst[c * 128] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                        }
                        part[kPartHalfWords + row] = bad ? (t_first == 0 ? 0.f : -INFINITY) : m_run;
                        part[kPartHalfWords + kMaxB + row] = bad ? (t_first == 0 ? 1.f : 0.f) : l_run;
                    }
                }
                ++seg;
            }
        }
    }

    // ---- teardown
    if constexpr (kCluster) {
        // merge of the cluster's partials: this CTA takes its share of the rows, a thread 16 columns of a row
        //   M = max m_p,  L = sum l_p 2^(m_p - M),  out = sum_p 2^(m_p - M) l_p (O/l)_p / L
        // (one warp a scheduler and some 300 dependent instructions: all arithmetic that needs no partial stands in front
        // of the barrier, and every load is unconditional -- a part that is not there is read from the first one, which
        // always is, and weighs nothing.  Partials in the CTAs' shared memory, read by ld.shared::cluster, were slower than
        // through L2: 15.65 against 14.4 us a call at 32 heads and 2k keys, 24.8 against 22.5 at 40 heads and 4k.)
        const int mt = kGrouped ? head / Hkv : 0, hk = head - mt * Hkv;
        const int rows = min(nb, nodes_of(n_nodes, 0, B) - mt * nb) * g;
        const bool split = T_all > 1 && rows > 0;          // (a single tile was written by the CTA that had it)
        const int r0 = rows * rank / cluster, n_rows = split ? rows * (rank + 1) / cluster - r0 : 0;
        int task = threadIdx.x;
        int u = n_rows > 0 ? task / n_rows : 0, row = r0 + task - u * n_rows;   // neighbouring threads: neighbouring rows
        const bool all_parts = T_all >= cluster;
        __syncwarp();
        tc_fence_before();
        cluster_sync();                                    // the head's partials are complete in the workspace (L2)
        for (; task < n_rows * 8;) {
            const float* at_m = partials + (size_t)head * cluster * kUmmaPartFloats + kPartHalfWords + row;
            const uint4* at_x = reinterpret_cast<const uint4*>(partials + (size_t)head * cluster * kUmmaPartFloats) + 2 * u * 128 + row;
            float M_run = -INFINITY, L_run = 0.f, acc[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) acc[c] = 0.f;
            for (int pb = 0; pb < cluster; pb += kCombineRound) {
                float mp[kCombineRound], lp[kCombineRound];
                uint4 x[kCombineRound][2];
                bool use[kCombineRound];
#pragma unroll
                for (int q = 0; q < kCombineRound; ++q) {
                    const int p = pb + q;
                    use[q] = p < cluster && (all_parts || rank_start(p + 1) > rank_start(p));
                    const size_t peer = use[q] ? p : 0;
                    const float* pm = at_m + peer * kUmmaPartFloats;
                    const uint4* px = at_x + peer * (kUmmaPartFloats / 4);
                    mp[q] = __ldcg(pm);
                    lp[q] = __ldcg(pm + kMaxB);
                    x[q][0] = __ldcg(px);
                    x[q][1] = __ldcg(px + 128);
                }
#pragma unroll
                for (int q = 0; q < kCombineRound; ++q)
                    if (!use[q]) { mp[q] = -INFINITY; lp[q] = 0.f; }
                merge_round(mp, lp, x, M_run, L_run, acc);
            }
            const int i_local = kGrouped ? row / g : row;
            const size_t at = (size_t)(mt * nb + i_local) * H + hk * g + (row - i_local * g);
            store_merged(out + at * kHeadDim + 16 * u, acc, L_run);
            if (lse && u == 0) lse[at] = (M_run + log2f(L_run)) * kLn2;
            task += kThreads;
            u = task / n_rows; row = r0 + task - u * n_rows;
        }
    } else {
        __syncwarp();
        tc_fence_before();
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// bf16 queries [rows][Hkv][g][128] -> 4-D map, box = 64 x g x 1 x box_rows: the g query heads of one key/value
// head for box_rows consecutive nodes, landing as rows (node, member) of one 128-byte-swizzled tile
bool make_q_map(void* fn, CUtensorMap* map, const void* base, int64_t rows, int Hkv, int g, int box_rows) {
    cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)g, (cuuint64_t)Hkv, (cuuint64_t)rows};
    cuuint64_t strides[3] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)g * kHeadDim * 2, (cuuint64_t)Hkv * g * kHeadDim * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)g, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = reinterpret_cast<EncodeTiledFn>(fn)(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base),
                                                     dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// bf16 tensor [rows][H][128] -> 3-D map, box = 64 x 1 x box_rows, 128-byte swizzle, zero fill out of bounds
bool make_map(void* fn, CUtensorMap* map, const void* base, int64_t rows, int H, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)H, (cuuint64_t)rows};
    cuuint64_t strides[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)H * kHeadDim * 2};
    cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = reinterpret_cast<EncodeTiledFn>(fn)(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base),
                                                     dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace

// Self-test of the bounded-wait path: one warp waits on a barrier that nothing ever completes, with a short
// limit.  The wait must give up, set GOOSE_ST_TIMEOUT in status[0] and let the kernel return normally, the same way
// a stalled pipeline of the attention kernel would.  Nothing here can hang: the only loop is the bounded wait.
__global__ void __launch_bounds__(32)
bounded_wait_selftest_kernel(int32_t* __restrict__ status, long long limit_cycles, int32_t* __restrict__ result) {
    __shared__ Header hd;
    if (threadIdx.x == 0) {
        mbar_init(&hd.pv_done, 1);
        hd.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    bool ok = true;
    if (threadIdx.x == 0) ok = mbar_wait_limit(&hd, &hd.pv_done, 0, status, limit_cycles);   // never completes
    __syncwarp();
    // the other lanes see the abort flag at once, as the other roles of the attention kernel would
    if (threadIdx.x != 0) ok = mbar_wait_limit(&hd, &hd.pv_done, 0, status, limit_cycles);
    // the shared primitive the top-k kernel waits with: 1 (aborted) with the raised flag, 2 (timed out) with a clear one
    __shared__ volatile int no_flag;
    if (threadIdx.x == 1) no_flag = 0;
    __syncwarp();
    int bad = 0;
    if (threadIdx.x == 1) {
        bad |= mbar_wait_bounded(&hd.pv_done, 0, limit_cycles, &hd.abort_flag) != 1;
        bad |= mbar_wait_bounded(&hd.pv_done, 0, limit_cycles, &no_flag) != 2;
        result[0] = (ok ? 1 : 0) | (bad ? 2 : 0);          // 0 expected: every wait reported failure, the kernel returns
    }
}

cudaError_t launch_bounded_wait_selftest(goose_ctx* c, long long limit_cycles, int32_t* result, cudaStream_t st) {
    bounded_wait_selftest_kernel<<<1, 32, 0, st>>>(c->status, limit_cycles, result);
    c->launches++;
    return cudaGetLastError();
}

namespace {
typedef void (*UmmaKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const int64_t*, const int32_t*, const int32_t*,
                           const int32_t*, int, int, int, int, int, int, uint32_t, int, int64_t, float, float*, int32_t*,
                           __nv_bfloat16*, float*);
UmmaKernel umma_kernel(bool grouped, bool counts, bool cluster) {
    if (cluster) return grouped ? (counts ? tree_attn_umma_kernel<true, true, true> : tree_attn_umma_kernel<true, false, true>)
                                : (counts ? tree_attn_umma_kernel<false, true, true> : tree_attn_umma_kernel<false, false, true>);
    return grouped ? (counts ? tree_attn_umma_kernel<true, true, false> : tree_attn_umma_kernel<true, false, false>)
                   : (counts ? tree_attn_umma_kernel<false, true, false> : tree_attn_umma_kernel<false, false, false>);
}
}  // namespace

cudaError_t init_umma_kernel(goose_ctx* c) {
    for (int i = 0; i < 8; ++i) {
        cudaError_t e = cudaFuncSetAttribute(umma_kernel(i & 1, i & 2, i & 4), cudaFuncAttributeMaxDynamicSharedMemorySize, kUmmaSmem);
        if (e != cudaSuccess) return e;
    }
    // how many clusters of each size the device holds at once (its SMs come in groups of unequal size)
    for (int n = 2; n <= kMaxCluster; ++n) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(n * c->num_sms); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kUmmaSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = n; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int m = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&m, umma_kernel(true, true, true), &cfg);
        if (e != cudaSuccess) return e;
        c->max_clusters[n] = m;
    }
    return cudaSuccess;
}

cudaError_t init_merge_kernel() {
    return load_kernels({(const void*)tree_attn_combine_kernel<false, false>, (const void*)tree_attn_combine_kernel<false, true>,
                         (const void*)tree_attn_combine_kernel<true, false>, (const void*)tree_attn_combine_kernel<true, true>});
}

int auto_attn_impl(const goose_ctx* c, int S, int B, int H) {
    (void)S; (void)H;
    (void)B;
    // the tcgen05 kernel wins at every tree size measured (B = 16: 15.8 us vs 31 us on the tiny workload);
    // the mma.sync kernel remains as the path for drivers that cannot encode tensor maps and on request
    return c->encode_tiled ? GOOSE_ATTN_UMMA : GOOSE_ATTN_MMA;
}

// One sequence: a cluster per head, the largest (of at most 8 CTAs) that the device holds one of per head at once (in a step with a
// long top-k a smaller one where that ends both earlier: see step_split()) -- where
// the SMs that this leaves out cost less than the merge kernel and the second segments that it saves.  What they cost grows
// with lost = tiles / n - heads * tiles / SMs, the tiles that the longest CTA has more than an equal share; what is saved
// depends on what else the launches do, so there are three kinds of call.  ctx_len[] is device data: the tiles are bounded
// by the rows of the cache, so that a long prefix never meets the slower form -- and a short one in a cache with many spare
// rows does not meet the faster one.  us, persistent -> clusters, (lost):
// the attention alone saves the merge kernel: 4.4, and no clusters of two
//   32 heads (n = 4) 2k (0.6) 16.1 -> 13.8, 16k (4.4) 51.5 -> 49.0;     40 heads (n = 3) 4k (2.1) 23.6 -> 22.7, 8k (4.1) 36.2 -> 35.2
//   52 heads (n = 2) 1k (1.3) 14.7 -> 15.5, 2k (2.5) 18.9 -> 20.4;      8 heads (n = 8) 4k (2.3) 15.8 -> 12.6, 12k (6.9) 21.7 -> 22.0
//   two to four M tiles a key/value head, 3.5:  16 heads (n = 6) 3k (1.4) 14.5 -> 12.5,
//   6k (2.8) 18.5 -> 17.6, 8k (3.8) 20.5 -> 20.4, 12k (5.7) 24.4 -> 27.2;   32 heads over 8 (n = 4) 16k (4.4) 43.5 -> 45.9
// a step whose top-k takes more than an item an SM, or the log-sum-exp too, has that beside the clusters: 4.4, and 3 for two
//   32 heads, 80 rows 16k (4.4) 55.3 -> 51.2;   40 heads 8k (4.1) 40.8 -> 39.2;   52 heads 2k (2.5) 25.9 -> 23.9, 3k (3.7) 29.7 -> 29.4,
//   4k (4.9) 33.5 -> 34.0;   8 heads, 32 rows 6k (3.5) 20.6 -> 19.3, 12k (6.9) 24.2 -> 26.0;   16 heads, 60 rows of 128256 8k (3.8) 31.7 -> 25.6
// any other step hides its top-k in the persistent form's ragged end and has the merge in its last launch: less is saved, by
// number of CTAs and of parts a head (the merge of 74 parts is slow)
//   52 heads 512 (0.7) 17.1 -> 18.9: no clusters of two;   40 heads 512 (0.3) 16.0 -> 15.0, 768 (0.4) 17.0 -> 16.7, 1k (0.6) 16.9 -> 17.7,
//   4k (2.1) 26.6 -> 27.2: 0.5 with three;   32 heads 2k (0.6) 18.7 -> 17.9, 8k (2.2) 33.1 -> 32.5, 14 heads (n = 8) 2k (0.5) 16.6 -> 15.7,
//   4k (1.0) 18.2 -> 18.1, 8k (2.0) 22.5 -> 22.5, 12k (3.0) 26.3 -> 26.9: 1.5 on 70 % of the SMs or more;   8 heads 4k (2.3) 17.7 -> 16.9,
//   6k (3.5) 19.0 -> 19.4 (19.7 -> 18.6 where no draft token is accepted), 16 heads 2k (1.0) 16.1 -> 15.0, 4k (1.9) 18.0 -> 18.3,
//   8k (3.8) 22.7 -> 23.8: 3.5
// up to four heads, whatever the call: the merge of 37 parts a head and more is slow
//   2 heads, call / step / with harvest 2k (1.9) 26.0 -> 9.6 / 24.0 -> 13.5 / 24.1 -> 13.8, 8k (7.2) 30.3 -> 16.5 / 32.9 -> 20.5 / 33.0 -> 20.6,
//   12k (10.8) 28.4 -> 20.9 / 26.8 -> 25.0 / 28.4 -> 24.8, 16k (14.4) 28.7 -> 25.3 / 27.8 -> 29.4 / 29.1 -> 29.6: 10, and one head has more to win
//   4 heads, tree of 60  2k (1.7) 17.3 -> 10.3 / 18.6 -> 13.9 / 21.6 -> 14.0, 6k (4.8) 19.7 -> 14.9 / 20.8 -> 18.5 / 22.2 -> 18.7,
//   8k (6.4) 19.8 -> 17.1 / 21.8 -> 20.8 / 23.0 -> 21.0, 10k (7.7) 20.6 -> 18.8 / 21.7 -> 22.4 / 23.0 -> 22.4: 6
int attn_heads(int B, int H, int Hkv) {
    const int g = H / Hkv, nb = B * g <= kTile ? B : kTile / g;
    return (B + nb - 1) / nb * Hkv;
}
bool attn_cluster_fits(const goose_ctx* c, int n, int S, int B, int H, int Hkv, int64_t kv_rows, int step) {
    const int Hw = attn_heads(B, H, Hkv);
    if (S != 1 || n < 2 || n > kMaxCluster) return false;   // (several may differ in length by any factor)
    if (c->max_clusters[n] < Hw || Hw * n > c->num_sms || (n == 2 && step != 2)) return false;
    const int64_t tiles = (kv_rows + kTile - 1) / kTile;
    int line = n == 2 ? 30 : Hw <= 2 ? 100 : Hw <= 4 ? 60 : 44;   // tenths of a tile
    if (Hw > Hkv && Hw > 4 && step == 0) line = 35;               // several M tiles a head: K/V come from L2, idle SMs cost their share
    if (step == 1 && Hw > 4) line = n == 3 ? 5 : 10 * Hw * n >= 7 * c->num_sms ? 15 : 35;
    return tiles * (c->num_sms - Hw * n) * 10 <= (int64_t)line * n * c->num_sms;
}
int attn_cluster(const goose_ctx* c, int S, int B, int H, int Hkv, int64_t kv_rows, int step) {
    const int Hw = attn_heads(B, H, Hkv);
    int n = 1;
    for (int i = 2; i <= kMaxCluster; ++i)
        if (c->max_clusters[i] >= Hw && Hw * i <= c->num_sms) n = i;
    return attn_cluster_fits(c, n, S, B, H, Hkv, kv_rows, step) ? n : 1;
}

cudaError_t launch_tree_attn_umma(goose_ctx* c, const __nv_bfloat16* q, const __nv_bfloat16* kc,
                                  const __nv_bfloat16* vc, int64_t kv_rows, const int64_t* row_off,
                                  const int32_t* ctx_len, const int32_t* parent, const int32_t* n_nodes, int S, int B, int H,
                                  int Hkv, float scale, __nv_bfloat16* out, float* lse, cudaStream_t st,
                                  CombinePlan* defer_merge, int cluster) {
    if (defer_merge) defer_merge->valid = false;
    if (!c->encode_tiled) return cudaErrorNotSupported;
    if (S == 0) return cudaSuccess;
    const int g = H / Hkv;                              // query heads per key/value head (validated by the caller)
    const int nb = B * g <= kTile ? B : kTile / g;      // nodes per M tile
    const int n_mt = (B + nb - 1) / nb;
    CUtensorMap mq, mk, mv;
    if (!make_q_map(c->encode_tiled, &mq, q, (int64_t)S * B, Hkv, g, nb) ||
        !make_map(c->encode_tiled, &mk, kc, kv_rows, Hkv, kTile) ||
        !make_map(c->encode_tiled, &mv, vc, kv_rows, Hkv, kTile))
        return cudaErrorInvalidValue;
    const int Hw = n_mt * Hkv;
    if (cluster == 0) cluster = attn_cluster(c, S, B, H, Hkv, kv_rows, 0);
    int grid = cluster > 1 ? Hw * cluster : c->num_sms;
    if (2 * grid > c->n_slots) grid = c->n_slots / 2;
    const int divisor = cluster > 1 ? cluster : grid;   // the one that the form needs on the device
    const uint32_t g_magic = (uint32_t)((0x100000000ull + divisor - 1) / divisor);
    const bool grouped = g > 1;
    const bool counts = n_nodes != nullptr;
    cudaError_t e = launch_pdl_cluster(umma_kernel(grouped, counts, cluster > 1), dim3(grid), dim3(kThreads), cluster, kUmmaSmem,
                                       st, mq, mk, mv, row_off, ctx_len, parent, n_nodes, S, B, H, Hkv, g, nb, g_magic, cluster,
                                       kv_rows, scale * kLog2e, c->partials, c->status, out, lse);
    c->launches++;
    if (e != cudaSuccess || cluster > 1) return e;          // (a cluster merges its head itself)
    CombineArgs ca;
    ca.ctx_len = ctx_len; ca.n_nodes = n_nodes; ca.S = S; ca.B = B; ca.H = H; ca.Hkv = Hkv; ca.g = g; ca.nb = nb;
    ca.G = grid; ca.G_magic = g_magic; ca.Hw = Hw; ca.kv_rows = (int)kv_rows; ca.partials = c->partials; ca.out = out; ca.lse = lse;
    const int row_groups = (nb * g + 31) / 32;
    if (defer_merge) {                                  // the caller runs the merge as a role of a later launch
        defer_merge->args = ca; defer_merge->row_groups = row_groups; defer_merge->grouped = grouped;
        defer_merge->valid = true;
        return cudaSuccess;
    }
    auto merge_kernel = grouped ? (counts ? tree_attn_combine_kernel<true, true> : tree_attn_combine_kernel<true, false>)
                                : (counts ? tree_attn_combine_kernel<false, true> : tree_attn_combine_kernel<false, false>);
    e = launch_pdl(merge_kernel, dim3(row_groups, ca.Hw, S), dim3(kCombineThreads), 0, st, ca);
    c->launches++;
    return e;
}

}  // namespace goose
