// Per-node argmax and top-k over bf16 logits (Algorithm 3 step 2; batched top-K harvest of App. C.1).
//
// A row is cut into equal chunks of at most 32768 elements; the (row, chunk) items, in row-major order, are dealt in
// contiguous ranges to a persistent grid of one CTA per SM.  The exact order is carried by 32-bit keys
//     (order-preserving 16-bit image of the bf16 value) << 16 | (0xFFFF - index_in_chunk)
// so "largest key" is "largest value, lowest index on ties", all keys are distinct, and a key carries its own index.
// Building a key costs several instructions per element, so keys are built only for candidates: elements not below T, the
// k-th largest of the 32 half-warp maxima of an item (at least k elements are >= T, hence the chunk's k best are among
// them; about ten of 32768 qualify).  Roles, coupled by mbarriers alone (no CTA-wide barrier):
//   control warp (1)     streams the items into a ring of three 64 KB shared-memory stages with bulk asynchronous copies
//                        (cp.async.bulk), ranks an item's candidates, merges the chunks of a row, writes the results
//   data warps (16)      64 values per thread into registers: thread maxima with packed-bf16 max, half-warp maxima with
//                        redux.sync.  With the log-sum-exp they also sum the exponentials relative to the largest value
//                        of the warp's first sweep, eight elements at a time behind their load, so that one warp's
//                        exponentials cover another's loads and maxima
//   collector warps (4)  T by rank counting (every lane counts the keys above its own: independent compares instead of k
//                        dependent reduction rounds); the threads whose maximum is >= T; keys of their elements >= T
// What bounds it: the stream (64 KB an item and SM: 1.47 us at the copy peak) and, with the log-sum-exp, the 32768
// exponentials of an item (2048 cycles of the special-function units).  The selection is a chain of some 500 dependent
// instructions on few warps (2000 to 4000 cycles by a clock trace); behind CTA-wide barriers, with every warp waiting for
// it, it was a third to half of an item's time.  Call times, one set of
// 1024-thread CTAs with three barriers an item -> these roles: 1500 x 32000 25.9 -> 19.2 us, with log-sum-exp and scatter
// 45.8 -> 26.6; 1024 x 32000 22.0 -> 14.5; 128 x 128256 11.7 -> 9.4; 480 x 32000 with counts and log-sum-exp 18.8 -> 12.7;
// one item a CTA (80 x 32000) 4.0 as before.  Measured and dropped: one barrier an item (23.1 and 40.8 us for 1500 rows),
// eight warps for the maxima and eight for the exponentials (39.4: two warps a scheduler do not fill the special-function
// units), a running maximum updated at every sweep (33.4: a redux.sync and a branch every eight elements).
// A quarter with many candidates (ties, as in a constant row) is cut with the k-th largest thread maximum instead and
// takes only the first k of the elements equal to it, so the list is bounded whatever the row holds.
// A row whose chunks are spread over several CTAs is finished by the last of those CTAs to arrive (arrival counter, no
// spinning).  Every mbarrier wait is bounded: when one runs out the CTA reports GOOSE_ST_TIMEOUT, drains its own copies in
// flight (bounded again) and returns.
#include <mutex>
#include <type_traits>

#include "goose_internal.cuh"
#include "topk_deal.cuh"

namespace goose {

constexpr int kTopkDataWarps = 16;
constexpr int kTopkCollectWarps = 4;
constexpr int kTopkDataThreads = kTopkDataWarps * 32;
constexpr int kTopkControlWarp = kTopkDataWarps + kTopkCollectWarps;
constexpr int kTopkThreads = (kTopkControlWarp + 1) * 32;    // 16 + 4 + 1 warps, and with a table one more
constexpr int kTopkPerThread = 64;                           // of a data thread: 8 x 128-bit shared-memory loads
static_assert(kTopkChunk == kTopkDataThreads * kTopkPerThread);
constexpr int kTopkSweep = kTopkDataThreads * 8;             // elements that the data threads load at once
constexpr int kTopkStages = 3;
constexpr int kTopkStageBytes = kTopkChunk * 2;              // 64 KB
// what an item hands from role to role lives in slot (item & 3): a slot comes back into use only after the control warp
// has finished its last item, because that warp issues item j + 4 behind finishing item j
constexpr int kTopkSlots = 4;
// a collector adds at most kTopkQuickList keys, or cuts with the k-th largest thread maximum T': fewer than k threads hold
// elements > T', 64 each, and of the elements equal to T' every collector takes at most k
constexpr int kTopkQuickList = 128;
constexpr int kTopkListCap = kMaxK * kTopkPerThread + kTopkCollectWarps * kMaxK + (kTopkCollectWarps - 1) * kTopkQuickList;
constexpr int kTableLoads = 8;                               // tokens a lane has in flight while it looks for a later row
constexpr int kTopkSmem = kTopkStages * kTopkStageBytes + kTopkSlots * kTopkListCap * 4;   // dynamic shared memory
constexpr long long kTopkWaitCycles = 2000000000ll;          // bound of every wait: about one second of SM clock
constexpr float kTopkLog2e = 1.4426950408889634f;
constexpr float kTopkLateMax = 11.f;                         // see the sums of exponentials: 11 log2(e) < 16
constexpr uint32_t kImageNegInf = 0x007Fu;                   // sortable16 of -inf

typedef unsigned long long u64;

__device__ __forceinline__ uint32_t sortable16(uint32_t bits) {
    bits &= 0xFFFFu;
    if (bits == 0x8000u) bits = 0;                           // -0.0 == +0.0
    return (bits & 0x8000u) ? (~bits & 0xFFFFu) : (bits | 0x8000u);
}

__device__ __forceinline__ float value_of_sortable16(uint32_t s) {
    uint32_t bits = (s & 0x8000u) ? (s ^ 0x8000u) : (~s & 0xFFFFu);
    return __uint_as_float(bits << 16);
}

__device__ __forceinline__ uint32_t bits_of_sortable16(uint32_t s) {
    return (s & 0x8000u) ? (s ^ 0x8000u) : (~s & 0xFFFFu);
}
__device__ __forceinline__ float topk_ex2(float x) {         // 2^x; results below 2^-126 are 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float float_of_sortable16(uint32_t s) { return __uint_as_float(bits_of_sortable16(s) << 16); }
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t w) { return *reinterpret_cast<__nv_bfloat162*>(&w); }
__device__ __forceinline__ uint32_t as_u32(__nv_bfloat162 v) { return *reinterpret_cast<uint32_t*>(&v); }

// largest 64-bit key of the warp: two 32-bit redux rounds (high words, then low words among the lanes that tie)
__device__ __forceinline__ u64 warp_max_u64(u64 v) {
    const uint32_t hi = (uint32_t)(v >> 32), lo = (uint32_t)v;
    const uint32_t mh = __reduce_max_sync(0xFFFFFFFFu, hi);
    const uint32_t ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? lo : 0u);
    return ((u64)mh << 32) | ml;
}


namespace {
__device__ __forceinline__ uint32_t topk_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void topk_mbar_init(u64* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(topk_smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void topk_mbar_arrive(u64* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(topk_smem_u32(bar)) : "memory");
}
// bit e of the result: element e of the eight in w is >= (or, with kStrict, >) the value in both halves of t (a NaN passes)
template <bool kStrict>
__device__ __forceinline__ uint32_t topk_above(const uint4& w, __nv_bfloat162 t) {
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t c = kStrict ? __hgtu2_mask(as_bf162(x[q]), t) : __hgeu2_mask(as_bf162(x[q]), t);
        m |= ((c & 1u) | ((c >> 15) & 2u)) << (2 * q);
    }
    return m;
}

// a walk over the rows that exist: rows of the call, or with node counts the rows of nodes that exist, numbered densely
template <bool COUNTS>
struct RowCursor {
    int row, chunk;            // current item: dense row number and chunk in it
    long long mem;             // the row's place in memory
    int s, left;               // its sequence, and the existing rows of that sequence from this one on
    __device__ __forceinline__ void seek(int w, int chunks, const int32_t* n_nodes, int S, int B) {
        row = w / chunks; chunk = w - row * chunks;
        mem = row; s = 0; left = 0;
        if (COUNTS) {
            int r = row;
            for (; s < S; ++s) {
                const int n = nodes_of(n_nodes, s, B);
                if (r < n) { mem = (long long)s * B + r; left = n - r; return; }
                r -= n;
            }
            mem = 0;                                         // behind the last row (a CTA without items): not used
        }
    }
    __device__ __forceinline__ void next(int chunks, const int32_t* n_nodes, int S, int B) {
        if (++chunk < chunks) return;
        chunk = 0; ++row; ++mem;
        if (COUNTS && --left == 0) {
            do ++s; while (s < S && (left = nodes_of(n_nodes, s, B)) == 0);
            mem = (long long)s * B;
        }
    }
};
}  // namespace

// LSE = true additionally returns the row's log-sum-exp (for the softmax scores of the harvest): the data warps sum
// exp(x - chunk max) over every element, chunks are merged like split softmax partials.  With a table (LSE without counts) the
// control warp also writes the row's ids and scores there, unless a later row has the same token: a scan of the later tokens, no
// atomics, by a warp of its own beside the item's stream.  1500 x 32000, a kernel behind this one -> here 26.0 -> 25.4 us (in the control
// warp, whose time the next copy waits for: 28.7); 16 tokens a lane in flight instead of 8: 2048 x 32000 31.5 -> 31.3, but
// 1500 x 128256 82.5 -> 84.8.
// COUNTS = false is the instantiation for n_nodes == NULL (the item list is known before the dependency wait)
// per, more, unit: TopkDeal.  The arguments with a table are 160 bytes: with 176 a launch took the host 0.4 us more (harvest calls 12.1 -> 12.6)
struct NoTable {};
template <bool LSE, bool COUNTS, class Table>
__global__ void __launch_bounds__(kTopkThreads + (std::is_same_v<Table, NoTable> ? 0 : 32), 1)
node_topk_kernel(const __nv_bfloat16* __restrict__ logits, int per, int more, int unit, int V, int64_t ldl, int k, int chunks,
                 int chunk_elems, int inputs_ready, u64* __restrict__ ws_cand, int32_t* __restrict__ row_counters,
                 int32_t* __restrict__ argmax, int32_t* __restrict__ ids, float* __restrict__ vals,
                 float* __restrict__ row_lse, float2* __restrict__ ws_lse, int32_t* __restrict__ status,
                 const int32_t* __restrict__ n_nodes, int S, int B, const Table table) {
    constexpr bool TABLE = !std::is_same_v<Table, NoTable>;
    extern __shared__ __align__(128) unsigned char s_stage[];   // kTopkStages x 64 KB, then the candidate lists
    __shared__ u64 s_full[kTopkStages];                  // the stage holds its item
    __shared__ u64 s_max_done[kTopkSlots], s_list_done[kTopkSlots];
    __shared__ __align__(16) uint32_t s_gmax[kTopkSlots][32];   // half-warp maxima as distinct keys: value image << 5 | 31 - index
    __shared__ __align__(16) unsigned short s_tmax[kTopkStages][kTopkDataThreads];   // thread maxima (value images)
    __shared__ float s_sum[kTopkSlots][kTopkDataWarps];   // sums of exponentials, and the images of what they are relative to
    __shared__ uint32_t s_sum_max[kTopkSlots][kTopkDataWarps];
    __shared__ int s_count[kTopkSlots];                  // length of the candidate list
    __shared__ unsigned short s_hold[kTopkCollectWarps][16];
    __shared__ __align__(16) uint32_t s_sel[32];         // rank-ordered keys of a selection
    __shared__ __align__(16) u64 s_m64[32];              // candidates of a 64-bit merge
    __shared__ u64 s_run[kMaxK];
    __shared__ u64 s_merge[kTopkMaxChunks * kMaxK];
    __shared__ int s_last;
    __shared__ int s_table_row[kTopkSlots];              // the table row that the item's logits row writes, -1: none
    __shared__ volatile int s_abort;
    uint32_t* const s_lists = reinterpret_cast<uint32_t*>(s_stage + kTopkStages * kTopkStageBytes);   // candidates' keys;
                                                         // entries 0..31 of a list are zero between items

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (!COUNTS) n_nodes = nullptr;
    const bool control = warp == kTopkControlWarp;

    if (control && lane == 0) {
        for (int i = 0; i < kTopkStages; ++i) topk_mbar_init(&s_full[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (tid < kTopkSlots) {
        topk_mbar_init(&s_max_done[tid], kTopkDataWarps);
        topk_mbar_init(&s_list_done[tid], kTopkCollectWarps + (TABLE ? 1 : 0));
        s_count[tid] = 0;
        if (tid == 0) s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1)
        for (int i = 0; i < kTopkSlots; ++i) s_lists[i * kTopkListCap + lane] = 0;
    // CTA c's items: the first `more` CTAs have `unit` more of them than the `per` that all have (32-bit arithmetic throughout: 64-bit
    // divisions in front of the first copy and barrier set-up by one thread had cost 0.5 us a call).  With node counts the rows
    // that exist are dealt below, item by item: whole rows where their share allows it were up to 15 % faster (121 of 240
    // rows of 128256 13.0 -> 11.4 us) and, by the divisions in front of the first copy, up to 4 % slower (176 of 200 rows of 262144 21.9 ->
    // 22.8, 359 of 480 rows of 32000 8.8 -> 9.1).
    const int G = gridDim.x;
    if (COUNTS) unit = 1;
    auto cta_start = [&](int c) { return c * per + min(c, more) * unit; };
    auto cta_of = [&](int w) { return w < more * (per + unit) ? w / (per + unit) : more + (w - more * (per + unit)) / per; };
    // inputs_ready: the caller guarantees that everything in front of the preceding kernel in the stream was complete when
    // this one could start, and that the preceding kernel touches neither the logits nor what this kernel writes (the
    // whole-step call: that kernel is the attention kernel, which lets its dependents start behind its own wait).  The
    // CTA then does all of its work beside that kernel and waits for it only before it ends, so that the completion of
    // this grid implies that kernel's.  (Waiting in front of the first result instead: CTAs with several items stood
    // still until the attention had ended, 1.6 us a step at 32 heads, 2k keys and 80 rows on 20 CTAs.)
    const bool wait_at_end = inputs_ready != 0;
    // the range is worked out ahead of the wait, while the kernel in front runs: behind it its arguments' first reads stood before the
    // first copy (rows of 32000: 128 rows 3.84 -> 3.75 us, harvest of 16 rows 4.90 -> 4.75)
    int w_begin = cta_start(blockIdx.x), n_local = cta_start(blockIdx.x + 1) - w_begin;
    asm volatile("" : "+r"(w_begin), "+r"(n_local));
    if (!wait_at_end) pdl_wait();
    pdl_trigger();
    // Per-sequence node counts (n_nodes != NULL; rows = S * B, row s * B + i belongs to node i of sequence s): rows of
    // nodes that do not exist are left out of the item list, so their logits are never read.  The list then runs over
    // the rows that exist, numbered densely (the cross-CTA scratch is indexed by that number).  n_nodes[] is an input
    // like the logits: it may be read ahead of the dependency wait.
    if (COUNTS && n_nodes) {
        int live = 0;
        for (int s = 0; s < S; ++s) live += nodes_of(n_nodes, s, B);
        const int items = live * chunks;
        per = items / G; more = items - per * G;
        w_begin = cta_start(blockIdx.x); n_local = cta_start(blockIdx.x + 1) - w_begin;
    }

    // control warp: the next item to stream; its first copies leave before the rest of the CTA is set up
    const unsigned short* lg = reinterpret_cast<const unsigned short*>(logits);
    RowCursor<COUNTS> in{};
    int issued = 0;
    // stream the next item into stage `issued` % kTopkStages (the copy is rounded up to 16 bytes, which stays inside the
    // row because ldl is a multiple of 8 elements)
    auto issue = [&]() {
        const int base = in.chunk * chunk_elems;
        const uint32_t bytes = ((uint32_t)min(chunk_elems, V - base) * 2u + 15u) & ~15u;
        const int st = issued % kTopkStages;
        if (lane == 0) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(topk_smem_u32(&s_full[st])), "r"(bytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(topk_smem_u32(s_stage + st * kTopkStageBytes)), "l"(lg + (size_t)in.mem * ldl + base), "r"(bytes),
                           "r"(topk_smem_u32(&s_full[st])) : "memory");
        }
        in.next(chunks, n_nodes, S, B);
        ++issued;
    };
    if (control) {
        in.seek(w_begin, chunks, n_nodes, S, B);
        while (issued < n_local && issued < kTopkStages) issue();
    }
    __syncthreads();

    // bounded wait for item j's hand-over in its slot; a wait that runs out raises the CTA's abort flag, which ends the
    // waits of all other warps
    auto slot_wait = [&](u64* bars, int j) -> bool {
        if (mbar_wait_bounded(&bars[j % kTopkSlots], (uint32_t)(j / kTopkSlots) & 1u, kTopkWaitCycles, &s_abort) == 0) return true;
        s_abort = 1;
        return false;
    };

    if (warp < kTopkDataWarps) {
        // ================================================================================ data warps
        int chunk = w_begin % chunks;
        for (int j = 0; j < n_local; ++j) {
            const int st = j % kTopkStages, slot = j % kTopkSlots;
            const unsigned char* sp = s_stage + st * kTopkStageBytes;
            const int n_valid = min(chunk_elems, V - chunk * chunk_elems);
            if (mbar_wait_bounded(&s_full[st], (uint32_t)(j / kTopkStages) & 1u, kTopkWaitCycles, &s_abort) != 0) {
                s_abort = 1;
                break;
            }
            // thread tid's 64 values: element (it, e) sits at chunk offset it * 4096 + tid * 8 + e; elements past the
            // chunk's end read as -inf
            auto trim = [&](uint4& w, int it) {
                const int off0 = it * kTopkSweep + tid * 8;
                if (off0 + 8 > n_valid) {
                    uint32_t y[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint32_t lo = (off0 + 2 * q < n_valid) ? (y[q] & 0xFFFFu) : 0xFF80u;
                        const uint32_t hi = (off0 + 2 * q + 1 < n_valid) ? (y[q] >> 16) : 0xFF80u;
                        y[q] = lo | (hi << 16);
                    }
                    w = make_uint4(y[0], y[1], y[2], y[3]);
                }
            };
            auto load = [&](int it) { return *reinterpret_cast<const uint4*>(sp + (size_t)(it * kTopkSweep + tid * 8) * 2); };
            auto load_trimmed = [&](int it) {
                uint4 w = load(it);
                trim(w, it);
                return w;
            };
            auto max8 = [&](const uint4& w) { return __hmax2(__hmax2(as_bf162(w.x), as_bf162(w.y)), __hmax2(as_bf162(w.z), as_bf162(w.w))); };
            auto image_max = [&](__nv_bfloat162 m) -> uint32_t {     // value image of the larger half
                const uint32_t lo = sortable16(as_u32(m) & 0xFFFFu), hi = sortable16(as_u32(m) >> 16);
                return lo > hi ? lo : hi;
            };
            __nv_bfloat162 m2;
            if (LSE) {
                // sum of exp(x - c), c = the largest value of the warp's first sweep; the control warp weights the sum with
                // the c it was taken with.  Elements past the end: 0.  Later sweeps may hold larger values: where one
                // is above c by more than 11 the sum is taken again, so that the exponents' arguments stay below 16 and their
                // rounding (2^-21) below that of the other steps.  (With a bound of 44 rows whose largest values come late were
                // off by up to 1.6e-6 instead of 0.8e-6; one warp that sums twice costs 2.4 us of 24 with 1500 x 32000 logits
                // that have one token 15 above the field each.)  Two lanes of packed fp32 arithmetic an instruction: the
                // issue slots, not the special-function units, would be the limit otherwise.
                auto add8 = [&](const uint4& w, u64 (&es)[2], float c) {
                    const u64 l2 = pack_f32x2(kTopkLog2e, kTopkLog2e), c2 = pack_f32x2(-c, -c);
                    const uint32_t y[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 t = unpack_f32x2(mul_f32x2(add_f32x2(pack_f32x2(__uint_as_float(y[q] << 16), __uint_as_float(y[q] & 0xFFFF0000u)), c2), l2));
                        es[q & 1] = add_f32x2(es[q & 1], pack_f32x2(topk_ex2(t.x), topk_ex2(t.y)));
                    }
                };
                const uint4 w0 = load_trimmed(0);
                m2 = max8(w0);
                uint32_t sum_max = __reduce_max_sync(0xFFFFFFFFu, image_max(m2));
                u64 es[2] = {0, 0};
                float c = sum_max == kImageNegInf ? 0.f : float_of_sortable16(sum_max);
                add8(w0, es, c);
#pragma unroll
                for (int it = 1; it < 8; ++it) {
                    const uint4 w = load_trimmed(it);
                    m2 = __hmax2(m2, max8(w));
                    add8(w, es, c);
                }
                const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, image_max(m2));
                if (wmax != kImageNegInf && (sum_max == kImageNegInf || float_of_sortable16(wmax) - c > kTopkLateMax)) {
                    sum_max = wmax;
                    c = float_of_sortable16(wmax);
                    es[0] = es[1] = 0;
                    for (int it = 0; it < 8; ++it) add8(load_trimmed(it), es, c);
                }
                const float2 e2 = unpack_f32x2(add_f32x2(es[0], es[1]));
                float sum = e2.x + e2.y;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
                if (lane == 0) { s_sum[slot][warp] = sum; s_sum_max[slot][warp] = sum_max; }
            } else {
                uint4 x[8];                                  // all loads first: nothing else hides their latency here
#pragma unroll
                for (int it = 0; it < 8; ++it) x[it] = load(it);
                if (n_valid < kTopkChunk) {
#pragma unroll
                    for (int it = 0; it < 8; ++it) trim(x[it], it);
                }
                m2 = max8(x[0]);
#pragma unroll
                for (int it = 1; it < 8; ++it) m2 = __hmax2(m2, max8(x[it]));
            }
            const uint32_t tmax = image_max(m2);             // this thread's maximum
            s_tmax[st][tid] = (unsigned short)tmax;
            const uint32_t h0 = __reduce_max_sync(0xFFFFFFFFu, lane < 16 ? tmax : 0u);
            const uint32_t h1 = __reduce_max_sync(0xFFFFFFFFu, lane < 16 ? 0u : tmax);
            if (lane < 2) s_gmax[slot][2 * warp + lane] = ((lane ? h1 : h0) << 5) | (uint32_t)(31 - 2 * warp - lane);
            __syncwarp();
            if (lane == 0) topk_mbar_arrive(&s_max_done[slot]);
            if (++chunk == chunks) chunk = 0;
        }
        if (wait_at_end) pdl_wait();
        return;
    }

    if (warp < kTopkDataWarps + kTopkCollectWarps) {
        // ================================================================================ collector warps
        const int c = warp - kTopkDataWarps;                 // looks after the data threads 128 c .. 128 c + 127
        int chunk = w_begin % chunks;
        for (int j = 0; j < n_local; ++j) {
            const int st = j % kTopkStages, slot = j % kTopkSlots;
            const unsigned short* sp = reinterpret_cast<const unsigned short*>(s_stage + st * kTopkStageBytes);
            const int n_valid = min(chunk_elems, V - chunk * chunk_elems);
            if (!slot_wait(s_max_done, j)) break;
            // T: lane l counts the half-warp maxima above the l-th (distinct keys); rank k-1 holds T
            const uint32_t v = s_gmax[slot][lane];
            const uint2 t4 = *reinterpret_cast<const uint2*>(&s_tmax[st][128 * c + 4 * lane]);   // four threads' maxima
            int rank = 0;
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                const uint4 w4 = *reinterpret_cast<const uint4*>(&s_gmax[slot][i]);
                rank += (w4.x > v) + (w4.y > v) + (w4.z > v) + (w4.w > v);
            }
            const uint32_t thr = __shfl_sync(0xFFFFFFFFu, v >> 5, __ffs(__ballot_sync(0xFFFFFFFFu, rank == k - 1)) - 1);
            // the threads that hold an element >= T: those whose maximum is (about ten of the item's 512)
            const uint32_t below = (1u << lane) - 1u;
            const uint32_t tm[4] = {t4.x & 0xFFFFu, t4.x >> 16, t4.y & 0xFFFFu, t4.y >> 16};
            int n_hold = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t b = __ballot_sync(0xFFFFFFFFu, tm[i] >= thr);
                const int at = n_hold + __popc(b & below);
                if (tm[i] >= thr && at < 16) s_hold[c][at] = (unsigned short)(128 * c + 4 * lane + i);
                n_hold += __popc(b);
            }
            __syncwarp();
            auto append = [&](uint32_t mask, int off) {      // keys of the elements off + (bits of mask)
                int at = mask ? atomicAdd(&s_count[slot], __popc(mask)) : 0;
                while (mask) {
                    const int o = off + __ffs(mask) - 1;
                    mask &= mask - 1;
                    if (at < kTopkListCap) s_lists[slot * kTopkListCap + at] = (sortable16(sp[o]) << 16) | (0xFFFFu - (uint32_t)o);
                    ++at;
                }
            };
            auto valid_mask = [&](int off) -> uint32_t {     // which of the eight elements from off on exist
                const int n = n_valid - off;
                return n >= 8 ? 0xFFu : n > 0 ? (1u << n) - 1u : 0u;
            };
            bool quick = n_hold <= 16;
            if (quick) {
                // four holders a round, eight lanes each: lane = (holder, sweep), eight elements per lane
                const __nv_bfloat162 t2 = as_bf162(bits_of_sortable16(thr) * 0x10001u);
                uint32_t masks = 0;
                for (int r = 0; 4 * r < n_hold; ++r) {
                    const int hi = 4 * r + (lane >> 3);
                    if (hi < n_hold) {
                        const int off = (lane & 7) * kTopkSweep + (int)s_hold[c][hi] * 8;
                        masks |= (topk_above<false>(*reinterpret_cast<const uint4*>(sp + off), t2) & valid_mask(off)) << (8 * r);
                    }
                }
                quick = __reduce_add_sync(0xFFFFFFFFu, __popc(masks)) <= kTopkQuickList;
                if (quick)
                    for (int r = 0; 4 * r < n_hold; ++r) {
                        const int hi = 4 * r + (lane >> 3);
                        const uint32_t m = (masks >> (8 * r)) & 0xFFu;
                        if (m) append(m, (lane & 7) * kTopkSweep + (int)s_hold[c][hi] * 8);
                    }
            }
            if (!quick) {
                // many candidates: T' = the k-th largest thread maximum (bisection over the 16-bit images), then this
                // quarter's elements in index order, all > T' and the first k of those equal to it
                const uint4* tp = reinterpret_cast<const uint4*>(&s_tmax[st][16 * lane]);
                const uint4 ta = tp[0], tb = tp[1];
                const uint32_t tw[8] = {ta.x, ta.y, ta.z, ta.w, tb.x, tb.y, tb.z, tb.w};
                uint32_t cut = 0;
                for (int b = 15; b >= 0; --b) {
                    const uint32_t cand = cut | (1u << b);
                    uint32_t n = 0;
#pragma unroll
                    for (int q = 0; q < 8; ++q) n += ((tw[q] & 0xFFFFu) >= cand) + ((tw[q] >> 16) >= cand);
                    if (__reduce_add_sync(0xFFFFFFFFu, n) >= (uint32_t)k) cut = cand;
                }
                const __nv_bfloat162 t2 = as_bf162(bits_of_sortable16(cut) * 0x10001u);
                int eq_left = k;
                for (int step = 0; step < 32; ++step) {
                    const int off = (step >> 2) * kTopkSweep + c * 1024 + (step & 3) * 256 + lane * 8;
                    const uint4 w4 = *reinterpret_cast<const uint4*>(sp + off);
                    const uint32_t valid = valid_mask(off);
                    const uint32_t gt = topk_above<true>(w4, t2) & valid;
                    uint32_t eq = topk_above<false>(w4, t2) & valid & ~gt;
                    if (eq_left > 0 && __any_sync(0xFFFFFFFFu, eq != 0)) {
                        int upto = __popc(eq);               // inclusive prefix over the lanes
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int u = __shfl_up_sync(0xFFFFFFFFu, upto, o);
                            if (lane >= o) upto += u;
                        }
                        int mine = min(__popc(eq), max(0, eq_left - (upto - __popc(eq))));
                        uint32_t keep = 0;
                        for (; mine > 0; --mine) { keep |= eq & -eq; eq &= eq - 1; }
                        eq_left -= __shfl_sync(0xFFFFFFFFu, upto, 31);
                        append(gt | keep, off);
                    } else {
                        append(gt, off);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) topk_mbar_arrive(&s_list_done[slot]);
            if (++chunk == chunks) chunk = 0;
        }
        if (wait_at_end) pdl_wait();
        return;
    }

    if constexpr (TABLE) if (warp > kTopkControlWarp) {
        // ================================================================================ table warp
        // which row of the table an item's logits row writes: a scan of the later rows' tokens beside the item's stream (an item's
        // arrival implies that its slot's last user is finished), for the items that end this CTA's part of a row alone -- nobody
        // reads the others' answer -- and up to the first later row with the token
        const int rows = cta_start(G) / chunks;
        int row = w_begin / chunks, chunk = w_begin - row * chunks;
        for (int j = 0; j < n_local; ++j) {
            if (mbar_wait_bounded(&s_full[j % kTopkStages], (uint32_t)(j / kTopkStages) & 1u, kTopkWaitCycles, &s_abort) != 0) {
                s_abort = 1;
                break;
            }
            int to = -1;
            if (chunk == chunks - 1 || j == n_local - 1) {
                const int tok = table.row_tok[row];
                bool stands = tok >= 0 && tok < table.table_rows;
                for (int r = row + 1; stands && r < rows; r += 32 * kTableLoads) {
                    bool later = false;
#pragma unroll
                    for (int u = 0; u < kTableLoads; ++u) later |= table.row_tok[min(r + u * 32 + lane, rows - 1)] == tok;
                    stands = !__any_sync(0xFFFFFFFFu, later);
                }
                if (stands) to = tok;
            }
            if (lane == 0) {
                s_table_row[j % kTopkSlots] = to;
                topk_mbar_arrive(&s_list_done[j % kTopkSlots]);
            }
            if (++chunk == chunks) { chunk = 0; ++row; }
        }
        if (wait_at_end) pdl_wait();
        return;
    }

    // ==================================================================================== control warp
    RowCursor<COUNTS> cur;                                   // the item being finished
    cur.seek(w_begin, chunks, n_nodes, S, B);
    // the current row's k best over the chunks walked so far (lane r: r-th 64-bit key value image << 32 | ~global index;
    // 0 = none) and its running log-sum-exp parts
    u64 run = 0;
    float run_m = -INFINITY, run_s = 0.f;
    bool part_starts_row = false;

    auto write_table = [&](int p, int32_t id, float val, float lse) {   // of the item in slot p, by the lanes below k
        if constexpr (TABLE) {
            const int at = s_table_row[p];
            if (at < 0) return;
            table.adj_ids[(size_t)at * k + lane] = id;
            table.adj_scores[(size_t)at * k + lane] = expf(val - lse);
        }
    };

    // rank the candidates of item i, merge them into the row's list, write what is complete
    auto finish_item = [&](int i) {
        const int p = i % kTopkSlots;
        uint32_t* list = s_lists + p * kTopkListCap;
        const int n_list = min(s_count[p], kTopkListCap);
        uint32_t mine = 0;                               // lane r: the chunk's r-th winner
        if (n_list <= 32) {
            // entries n_list..31 are zero: lane l ranks key l among the (distinct) keys
            const uint32_t c = list[lane];
            int rank = 0;
#pragma unroll
            for (int q = 0; q < 32; q += 4) {
                const uint4 w4 = *reinterpret_cast<const uint4*>(&list[q]);
                rank += (w4.x > c) + (w4.y > c) + (w4.z > c) + (w4.w > c);
            }
            __syncwarp();
            if (c != 0) s_sel[rank] = c;
            __syncwarp();
            mine = lane < min(k, n_list) ? s_sel[lane] : 0u;
        } else {
            for (int r = 0; r < k; ++r) {
                uint32_t m = 0;
                for (int q = lane; q < n_list; q += 32) m = list[q] > m ? list[q] : m;
                const uint32_t w = __reduce_max_sync(0xFFFFFFFFu, m);
                if (lane == r) mine = w;
                if (w != 0)
                    for (int q = lane; q < n_list; q += 32)
                        if (list[q] == w) list[q] = 0;
                __syncwarp();
            }
        }
        __syncwarp();
        list[lane] = 0;                                  // entries 0..31 are zero between items
        if (lane == 0) s_count[p] = 0;

        const int row = cur.row, chunk = cur.chunk, base = chunk * chunk_elems;
        const size_t out_row = (size_t)cur.mem;
        cur.next(chunks, n_nodes, S, B);
        float csum = 0.f;
        const float cmax = LSE ? float_of_sortable16(__reduce_max_sync(0xFFFFFFFFu, s_gmax[p][lane]) >> 5) : 0.f;
        if (LSE) {
            // warp w's sum is relative to its c_w: weight exp(c_w - cmax)
            if (lane < kTopkDataWarps) {
                const uint32_t m = s_sum_max[p][lane];
                if (m != kImageNegInf) csum = s_sum[p][lane] * topk_ex2((float_of_sortable16(m) - cmax) * kTopkLog2e);   // else: -inf alone
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) csum += __shfl_xor_sync(0xFFFFFFFFu, csum, o);
        }
        if (chunks == 1) {                               // the chunk is the row: write it out
            if (lane < k) {
                const int32_t id = (int32_t)(0xFFFFu - (mine & 0xFFFFu));
                ids[out_row * k + lane] = id;
                if (vals) vals[out_row * k + lane] = value_of_sortable16(mine >> 16);
                if (lane == 0) argmax[out_row] = id;
                if constexpr (TABLE) write_table(p, id, value_of_sortable16(mine >> 16), cmax + logf(csum));
            }
            if (LSE && lane == 0) row_lse[out_row] = cmax + logf(csum);
            return;
        }
        const bool part_begins = (i == 0) || (chunk == 0);
        const bool part_ends = (i == n_local - 1) || (chunk == chunks - 1);
        if (part_begins) part_starts_row = (chunk == 0);
        // this chunk's winners as 64-bit keys of the row
        const u64 ck = mine ? (((u64)(mine >> 16) << 32) | (u64)(0xFFFFFFFFu - (uint32_t)(base + (int)(0xFFFFu - (mine & 0xFFFFu))))) : 0ull;
        if (part_begins) {
            run = lane < k ? ck : 0ull;
            run_m = cmax; run_s = csum;
        } else {
            // merge the running list and the chunk's (k keys each, all distinct): lanes 0..15 offer the running
            // list, lanes 16..31 the chunk's, every lane counts the keys above its own
            const u64 shifted = __shfl_sync(0xFFFFFFFFu, ck, (lane + 16) & 31);   // lane 16 + r <- ck of lane r
            const u64 cand = lane < 16 ? (lane < k ? run : 0ull) : (lane - 16 < k ? shifted : 0ull);
            s_m64[lane] = cand;
            if (lane < kMaxK) s_run[lane] = 0;
            __syncwarp();
            int rank = 0;
#pragma unroll
            for (int q = 0; q < 32; q += 2) {
                const ulonglong2 w2 = *reinterpret_cast<const ulonglong2*>(&s_m64[q]);
                rank += (w2.x > cand) + (w2.y > cand);
            }
            if (cand != 0 && rank < k) s_run[rank] = cand;
            __syncwarp();
            run = lane < k ? s_run[lane] : 0ull;
            __syncwarp();
            if (LSE) {
                const float M = fmaxf(run_m, cmax);          // -inf: nothing but -inf so far, both sums are 0
                if (M != -INFINITY) run_s = run_s * expf(run_m - M) + csum * expf(cmax - M);
                run_m = M;
            }
        }
        if (!part_ends) return;
        u64 win = run;
        float fin_m = run_m, fin_s = run_s;
        if (!(part_starts_row && chunk == chunks - 1)) {
            // the row's chunks are spread over several CTAs: CTAs c_first..c_last each hold one part
            const int c_first = cta_of(row * chunks), c_last = cta_of(row * chunks + chunks - 1);
            const int n_parts = c_last - c_first + 1, slot = (int)blockIdx.x - c_first;
            u64* dst = ws_cand + ((size_t)row * chunks + slot) * kMaxK;
            if (lane < k) dst[lane] = run;
            if (LSE && lane == 0) ws_lse[(size_t)row * chunks + slot] = make_float2(run_m, run_s);
            __threadfence();
            __syncwarp();
            if (lane == 0) {
                const int old = atomicAdd(&row_counters[row], 1);
                s_last = (old == n_parts - 1);
            }
            __syncwarp();
            if (!s_last) return;
            __threadfence();
            const u64* src = ws_cand + (size_t)row * chunks * kMaxK;
            const int n = n_parts * k;
            if (n <= 32) {
                const u64 cand = lane < n ? __ldcg(src + (size_t)(lane / k) * kMaxK + (lane % k)) : 0ull;
                s_m64[lane] = cand;
                if (lane < kMaxK) s_run[lane] = 0;
                __syncwarp();
                int rank = 0;
#pragma unroll
                for (int q = 0; q < 32; q += 2) {
                    const ulonglong2 w2 = *reinterpret_cast<const ulonglong2*>(&s_m64[q]);
                    rank += (w2.x > cand) + (w2.y > cand);
                }
                if (cand != 0 && rank < k) s_run[rank] = cand;
                __syncwarp();
                win = lane < k ? s_run[lane] : 0ull;
                __syncwarp();
            } else {
                for (int q = lane; q < n; q += 32) s_merge[q] = __ldcg(src + (size_t)(q / k) * kMaxK + (q % k));
                __syncwarp();
                win = 0;
                for (int r = 0; r < k; ++r) {
                    u64 m = 0;
                    for (int q = lane; q < n; q += 32) m = s_merge[q] > m ? s_merge[q] : m;
                    const u64 w = warp_max_u64(m);
                    if (lane == r) win = w;
                    if (w != 0)
                        for (int q = lane; q < n; q += 32)
                            if (s_merge[q] == w) s_merge[q] = 0;
                    __syncwarp();
                }
            }
            if (lane == 0) row_counters[row] = 0;        // ready for the next launch
            if (LSE && lane == 0) {
                float M = -INFINITY;
                for (int c = 0; c < n_parts; ++c) M = fmaxf(M, __ldcg(&ws_lse[(size_t)row * chunks + c]).x);
                float sum = 0.f;
                for (int c = 0; c < n_parts; ++c) {
                    const float2 ms = __ldcg(&ws_lse[(size_t)row * chunks + c]);
                    if (ms.x != -INFINITY) sum += ms.y * expf(ms.x - M);
                }
                fin_m = M; fin_s = sum;
            }
        }
        if (lane < k) {
            const int32_t id = (int32_t)(0xFFFFFFFFu - (uint32_t)(win & 0xFFFFFFFFull));
            ids[out_row * k + lane] = id;
            if (vals) vals[out_row * k + lane] = value_of_sortable16((uint32_t)(win >> 32));
            if (lane == 0) argmax[out_row] = id;
        }
        if (LSE && lane == 0) row_lse[out_row] = fin_m + logf(fin_s);
        if constexpr (TABLE) {                           // (parts of several CTAs: lane 0 merged them)
            const float lse = __shfl_sync(0xFFFFFFFFu, fin_m + logf(fin_s), 0);
            if (lane < k) write_table(p, (int32_t)(0xFFFFFFFFu - (uint32_t)(win & 0xFFFFFFFFull)), value_of_sortable16((uint32_t)(win >> 32)), lse);
        }
    };

    for (int j = 0; j < n_local; ++j) {
        const bool have = slot_wait(s_list_done, j);     // (implies the maxima and sums: the collectors waited for them)
        __syncwarp();                                    // every lane's clears of item j - 1's list stand before the copy that
                                                         // lets the slot's next user in (lane 0 alone issues it)
        if (have && issued < n_local) {                  // nobody reads item j's stage any more
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue();
        }
        if (!have) {
            // give up: report, wait (bounded) for the copies still in flight, return
            if (lane == 0) {
                if (status) atomicOr(status, GOOSE_ST_TIMEOUT);
                volatile int no_abort = 0;               // draining ignores the abort flag
                for (int jj = j; jj < issued; ++jj)
                    mbar_wait_bounded(&s_full[jj % kTopkStages], (uint32_t)(jj / kTopkStages) & 1u, kTopkWaitCycles, &no_abort);
            }
            break;
        }
        finish_item(j);
    }
    if (wait_at_end) pdl_wait();
}

namespace {
cudaError_t launch_topk_any(int num_sms, cudaStream_t st, const __nv_bfloat16* logits, int rows, int V, int64_t ldl, int k,
                            u64* ws, int32_t* counters, int32_t* argmax, int32_t* ids, float* vals, float* row_lse,
                            float2* ws_lse, int32_t* status, int inputs_ready, const int32_t* n_nodes = nullptr, int B = 0,
                            HarvestTable table = {}, bool beside = false) {
    const int S = (n_nodes && B > 0) ? rows / B : 0;
    // equal chunks (a multiple of 8 elements: every copy starts on 16 bytes), so that no item is a remainder
    const int chunks = topk_chunks(V);
    const int chunk_elems = ((V + chunks - 1) / chunks + 7) & ~7;
    const TopkDeal deal = topk_deal(rows, chunks, num_sms, row_lse || beside, n_nodes != nullptr);   // (a row costs the context 1 KB of
                                                     // scratch a chunk: its items are far below 2^31)
    auto launch = [&](auto kernel, int threads, auto with) {
        return launch_pdl(kernel, dim3(deal.grid), dim3(threads), kTopkSmem, st, logits, deal.per, deal.more, deal.unit, V, ldl, k, chunks, chunk_elems,
                          inputs_ready, ws, counters, argmax, ids, vals, row_lse, ws_lse, status, n_nodes, S, B, with);
    };
    if (table.adj_ids) return launch(node_topk_kernel<true, false, HarvestTable>, kTopkThreads + 32, table);
    return launch(row_lse ? (n_nodes ? node_topk_kernel<true, true, NoTable> : node_topk_kernel<true, false, NoTable>)
                          : (n_nodes ? node_topk_kernel<false, true, NoTable> : node_topk_kernel<false, false, NoTable>), kTopkThreads, NoTable{});
}
}  // namespace


// per-device kernel attributes: the stage ring needs the opt-in shared-memory size
cudaError_t init_topk_kernel() {
    cudaError_t e = cudaSuccess;
    auto opt_in = [&](const void* fn) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTopkSmem);
    };
    opt_in((const void*)node_topk_kernel<false, false, NoTable>);  opt_in((const void*)node_topk_kernel<false, true, NoTable>);
    opt_in((const void*)node_topk_kernel<true, false, NoTable>);   opt_in((const void*)node_topk_kernel<true, true, NoTable>);
    return e;
}
cudaError_t init_table_kernel() {
    return cudaFuncSetAttribute(node_topk_kernel<true, false, HarvestTable>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTopkSmem);
}

cudaError_t launch_node_topk(goose_ctx* c, const __nv_bfloat16* logits, int rows, int V, int64_t ldl, int k,
                             int32_t* argmax, int32_t* ids, float* vals, float* row_lse, cudaStream_t st,
                             bool inputs_ready, const int32_t* n_nodes, int B, int max_ctas, HarvestTable table) {
    if (rows == 0) return cudaSuccess;
    cudaError_t e = launch_topk_any(max_ctas > 0 ? max_ctas : c->num_sms, st, logits, rows, V, ldl, k, c->topk_cand, c->row_counters, argmax, ids, vals,
                                    row_lse, reinterpret_cast<float2*>(c->topk_lse_ws), c->status, inputs_ready ? 1 : 0,
                                    n_nodes, B, table, max_ctas > 0);
    c->launches++;
    return e;
}


// ---------------------------------------------------------------------------------------------------
// goose_node_topk_static: the same kernel for callers that are not allowed to allocate device memory
// (a host that pre-plans all device memory and forbids cudaMalloc at run time, or code running where
// the allocator must not be entered).  The cross-chunk scratch lives in a file-scope device array that
// every GPU loading this library carries until the process exits.
constexpr int kStaticMaxRows = GOOSE_STATIC_TOPK_MAX_ROWS;
constexpr size_t kStaticCandWords = (size_t)kStaticMaxRows * kTopkMaxChunks * kMaxK;   // per (row, chunk) winners: 2 MiB
constexpr size_t kStaticCounterWords = kStaticMaxRows / 2;                             // int32 arrival counters: 8 KiB
static __device__ __align__(256) u64 g_static_topk[kStaticCandWords + kStaticCounterWords];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
u64* g_static_ptr[kMaxDevices] = {};                             // device address of g_static_topk, per device
int g_static_sms[kMaxDevices] = {};                              // SM count, per device
}  // namespace

}  // namespace goose

extern "C" int goose_node_topk_static(const void* logits, int rows, int V, int64_t ldl, int k,
                                      int32_t* argmax, int32_t* topk_ids, float* topk_vals, void* stream) {
    using namespace goose;
    if (!logits || !argmax || !topk_ids) return GOOSE_EINVAL;
    if (rows < 0 || rows > kStaticMaxRows) return GOOSE_EINVAL;          // beyond the static scratch
    if (V < 1 || V > GOOSE_MAX_V || ldl < V || (ldl & 7) != 0) return GOOSE_EINVAL;
    if ((reinterpret_cast<uintptr_t>(logits) & 15u) != 0) return GOOSE_EINVAL;
    if (k < 1 || k > GOOSE_MAX_K || k > V) return GOOSE_EINVAL;
    if (rows == 0) return GOOSE_OK;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return GOOSE_ECUDA;
    u64* scratch;
    int num_sms;
    {
        // In host code the name g_static_topk is only a handle for the runtime, not a device address:
        // resolve the address once per device, with that device current.
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_ptr[dev]) {
            u64* p = nullptr;
            int sms = 0;
            if (cudaGetSymbolAddress((void**)&p, g_static_topk) != cudaSuccess || !p) return GOOSE_ECUDA;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return GOOSE_ECUDA;
            if (init_topk_kernel() != cudaSuccess) return GOOSE_ECUDA;   // a function attribute, not an allocation
            g_static_sms[dev] = sms;
            g_static_ptr[dev] = p;
        }
        scratch = g_static_ptr[dev];
        num_sms = g_static_sms[dev];
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int chunks = topk_chunks(V);
    // the counters must start at zero; the array keeps whatever an earlier (possibly interrupted) call left
    int32_t* counters = reinterpret_cast<int32_t*>(scratch + kStaticCandWords);
    if (chunks > 1 && cudaMemsetAsync(counters, 0, sizeof(int32_t) * (size_t)rows, st) != cudaSuccess)
        return GOOSE_ECUDA;
    cudaError_t e = launch_topk_any(num_sms, st, static_cast<const __nv_bfloat16*>(logits), rows, V, ldl, k, scratch, counters,
                                    argmax, topk_ids, topk_vals, static_cast<float*>(nullptr), static_cast<float2*>(nullptr),
                                    static_cast<int32_t*>(nullptr), 0);
    return e == cudaSuccess ? GOOSE_OK : GOOSE_ECUDA;
}
