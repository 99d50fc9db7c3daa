// Pieces of the tensor-core attention path that two kernels share: the work partition of the persistent main kernel
// and the merge of its split-KV partials.  The merge runs either as a kernel of its own (goose_tree_attn) or as a block
// role of the step's last launch (goose_verify_step), where it overlaps the acceptance walk and the compaction instead
// of standing between the attention kernel and the top-k.
#pragma once

#include <cuda_fp16.h>

#include "goose_internal.cuh"

namespace goose {

constexpr int kTile = 128;                       // keys per tile
constexpr float kLn2 = 0.6931471805599453f;
constexpr int kCombineThreads = 256;
constexpr int kCombineRound = 4;                 // partials merged per load round of the merge
// split-KV partial of the main kernel: normalised O/l as fp16, uint4 [16 column groups of 8][128 rows] (32 KB, a warp's
// stores and the merge's loads are contiguous), then m[128], l[128] as fp32
constexpr int kPartHalfWords = 16 * 128 * 4;     // 32-bit words of the fp16 block
constexpr int kUmmaPartFloats = kPartHalfWords + 2 * kMaxB;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// ---------------------------------------------------------------- work partition (same code in every role)
// The arithmetic compiles for the host as well, where a test walks it over lengths that no kernel should meet.
//
// 64-bit division out of line.  The merge finds CTAs and their starts in a dozen places, each with such a division for lists of
// 2^31 / SMs items and more: a third of its code, fetched by every launch and reached by hardly any (step of 40 heads at 4k, with
// the merge beside walk and compaction: 25.8 -> 25.1 us; 52 heads at 8k 45.8 -> 45.3).
static __host__ __device__ __noinline__ long long div64(long long a, long long b) { return a / b; }
__host__ __device__ __forceinline__ uint32_t mul_hi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
struct Work {
    const int32_t* ctx_len;
    const int32_t* n_nodes;   // per-sequence node counts, or NULL (every tree has B nodes)
    int S, H, B, G;           // H = heads of the work list = M tiles x key/value heads (M-tile-major)
    int kv_rows;              // rows of the cache, see prefix()
    uint32_t G_magic;         // ceil(2^32 / G): division by G without the 20-instruction sequence
    long long total;          // all items
    int pad;                  // idle items in front of every head, see set_total
    bool small;               // total * (G + 1) fits 31 bits: 32-bit arithmetic (64-bit division is slow on the GPU)
    // ctx_len comes from device memory.  A negative value is treated as 0 (the tree rows alone), a prefix longer than the cache
    // as one of the whole cache: such a sequence is flagged and zero-filled, and its list stays one that every range, count and
    // division below is right for.
    __host__ __device__ __forceinline__ int prefix(int ctx) const { return min(max(ctx, 0), kv_rows); }
    // A sequence's keys are its prefix and the nodes its tree really has; a sequence without nodes (it has left the batch) has
    // no items.
    __host__ __device__ __forceinline__ int tiles_of(int ctx, int nn) const {
        return (int)(((uint32_t)prefix(ctx) + (uint32_t)nn + kTile - 1) / kTile);
    }
    __host__ __device__ __forceinline__ int tiles(int s) const {
        if (!n_nodes) return tiles_of(ctx_len[s], B);
        const int nn = nodes_of(n_nodes, s, B);
        return nn == 0 ? 0 : tiles_of(ctx_len[s], nn);
    }
    // items of a head of T tiles
    __host__ __device__ __forceinline__ int width(int T) const { return T > 0 ? T + pad : 0; }
    // A CTA that goes over from one head to the next pays for it (its epilogue and the next head's first softmax stand in
    // turn: 2 to 3 us), so a head starts with idle items that take as much of the CTA's range.  Two tiles' worth, from two tiles
    // a CTA on (a CTA whose whole share is idle items has no work, as one without a share).  Attention call with none / 1 / 2, us:
    // 8 x 32 heads, 333 to 6000 keys 69.7 / 61.5 / 57.7;  16 x 32 over 8, 1k to 8k 63.8 / 60.8 / 59.4;  4 x 16 over 2, 8k 29.5 / 28.4 / 27.9;
    // 2 x 32, 4k to 8k 42.5 / 40.3 / 40.0;  2 x 32 over 8, tree of 61, 1k to 5k 19.9 / 20.0 / 20.4;  52 heads 4k 27.4 / 26.4 / 27.2, 8k
    // 43.9 / 43.4 / 43.4.  In long streams a head switch hides behind the other CTAs' loads and the idle items cost as little:
    // 8 x 32, 16k 329.5 / 329.7 / 329.6, 16 x 32, 1k to 16k 389.2 / 389.7 / 389.1 (sustained 438 / 438 / 436).
    __host__ __device__ __forceinline__ void set_total(long long tile_count, int live) {
        pad = tile_count >= 2 * (long long)G ? 2 : 0;
        total = tile_count + (long long)pad * H * live;
        small = total * (G + 1) < 0x7FFFFFFFll;
    }
    __host__ __device__ __forceinline__ void init() {
        long long tot = 0;
        int live = 0;
        auto add = [&](int s) {
            const int T = tiles(s);
            tot += (long long)H * T;
            live += T > 0;
        };
        // (small without counts; with them unrolled, since two dependent loads a sequence would follow one another)
        if (n_nodes) for (int s = 0; s < S; ++s) add(s);
        else
#pragma unroll 1
            for (int s = 0; s < S; ++s) add(s);
        set_total(tot, live);
    }
    // the same by a whole warp from the tiles of up to 32 sequences, one a lane (has: the lane's sequence has any)
    __device__ __forceinline__ void init_lanes(int tiles, bool has) {
        set_total(H * (long long)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)tiles), __popc(__ballot_sync(0xFFFFFFFFu, has)));
    }
    // the same by a whole warp, lane s loading sequence s's length; returns the tiles of sequence `lane`
    __device__ __forceinline__ int init_warp(int lane) {
        const int mine = lane < S ? tiles(lane) : 0;
        long long sum = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)mine);
        int live = n_nodes ? __popc(__ballot_sync(0xFFFFFFFFu, mine > 0)) : S;
        for (int s0 = 32; s0 < S; s0 += 32) {
            const int more = s0 + lane < S ? tiles(s0 + lane) : 0;
            sum += __reduce_add_sync(0xFFFFFFFFu, (uint32_t)more);
            if (n_nodes) live += __popc(__ballot_sync(0xFFFFFFFFu, more > 0));
        }
        set_total(H * sum, live);
        return mine;
    }
    template <bool kCall = false>
    __host__ __device__ __forceinline__ long long cta_start(int c) const {
        if (!small) return kCall ? div64(total * c, G) : total * c / G;
        const uint32_t n = (uint32_t)total * (uint32_t)c, q = mul_hi(n, G_magic);   // exact or one too large (n < 2^31)
        return q * (uint32_t)G > n ? q - 1 : q;
    }
    __host__ __device__ __forceinline__ int cta_of(long long w) const {
        int c = small ? (int)(((uint32_t)w * (uint32_t)G) / (uint32_t)total) : (int)div64(w * G, total);
        if (c >= G) c = G - 1;
#pragma unroll 1
        while (c + 1 < G && cta_start<true>(c + 1) <= w) ++c;
#pragma unroll 1
        while (c > 0 && cta_start<true>(c) > w) --c;
        return c;
    }
};

// first tile of CTA r of the n CTAs (a cluster) that share a head of T tiles; rounded up, so that the last CTA, which has the
// masked tile, has no tile more than the others.  n_magic = ceil(2^32 / n): a division by a multiplication, exact for the
// T * 8 < 2^28 that Work::tiles_of() can give (the division itself stood in front of the first load: attention call 512 keys
// 8.51 -> 8.15, 1531 11.78 -> 11.42, 32 over 8 heads 3k 12.50 -> 12.10 us)
__host__ __device__ __forceinline__ int cluster_start(int T, int r, int n, uint32_t n_magic) {
    return (int)mul_hi((uint32_t)(T * r + n - 1), n_magic);
}

struct Cursor {               // walks items in order
    long long w;              // item index
    int s, h, t, T;
    __host__ __device__ __forceinline__ void seek(const Work& wk, long long w0) {
        long long off = 0;
        int ss = 0;
        int TT = wk.tiles(0);
        while (ss + 1 < wk.S && off + (long long)wk.H * wk.width(TT) <= w0) {
            off += (long long)wk.H * wk.width(TT);
            ++ss;
            TT = wk.tiles(ss);
        }
        s = ss; T = TT; w = w0;
        const long long rem = w0 - off;
        const int W = wk.width(TT);
        h = wk.small ? (int)((uint32_t)rem / (uint32_t)W) : (int)(rem / W);
        enter(wk, (int)(rem - (long long)h * W));
    }
    // at item v of the head: past the idle ones
    __host__ __device__ __forceinline__ void enter(const Work& wk, int v) {
        t = v - wk.pad;
        if (t < 0) { w -= t; t = 0; }
    }
    // the same by a whole warp for the common small batch: `mine` = tiles of sequence `lane` (Work::init_warp)
    __device__ __forceinline__ void seek_warp(const Work& wk, long long w0, int lane, int mine) {
        if (!wk.small || wk.S > 32) { seek(wk, w0); return; }
        w = w0;
        uint32_t rem = (uint32_t)w0;
        s = 0;
        if (wk.S > 1) {
            const uint32_t own = (uint32_t)wk.H * (uint32_t)wk.width(mine);
            uint32_t upto = own;                                 // items up to and with sequence `lane`
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, upto, o);
                if (lane >= o) upto += u;
            }
            s = __ffs(__ballot_sync(0xFFFFFFFFu, upto > rem)) - 1;   // (w0 < total: some lane has it)
            rem -= __shfl_sync(0xFFFFFFFFu, upto - own, s);
        }
        T = __shfl_sync(0xFFFFFFFFu, mine, s);
        const int W = wk.width(T);
        h = (int)__float2uint_rz(__fdividef((float)rem, (float)W));   // h < 2^16: off by one at most
        int v = (int)rem - h * W;
        if (v < 0) { --h; v += W; }
        if (v >= W) { ++h; v -= W; }
        enter(wk, v);
    }
    // is any of the items from here to `w_end` a tile?  (where a head's idle items were skipped there may be none)
    __host__ __device__ __forceinline__ bool any(long long w_end) const { return w < w_end; }
    // items of this head from here to its end, at most up to item `w_end` of the list; and past n of them
    __host__ __device__ __forceinline__ int run(long long w_end) const { return (int)min((long long)(T - t), w_end - w); }
    __host__ __device__ __forceinline__ void skip(const Work& wk, int n) {
        w += n; t += n;
        if (t == T) {
            t = 0; ++h; w += wk.pad;
            if (h == wk.H) {                              // next sequence that has any items
                h = 0; ++s;
                if (!wk.n_nodes) { if (s < wk.S) T = wk.tiles(s); }
                else while (s < wk.S && (T = wk.tiles(s)) == 0) ++s;
            }
        }
    }
};

// ---------------------------------------------------------------- merge of the split-KV partials
// One call handles 32 rows (rg = row group) of head h (a head of the work list = M tile x key/value head) of sequence s
// with 256 threads.  A head that one CTA of the main kernel covered entirely was written directly and is skipped; any
// other is the merge of its CTAs' partials:
//   M = max m_p,  L = sum l_p 2^(m_p - M),  out = sum_p 2^(m_p - M) O_p / L.
// Lane <-> row (coalesced float4 loads of the transposed partial layout), warp <-> 16 output columns.
// The function contains the caller's dependency wait (pdl_wait / pdl_trigger): everything in front of it needs only
// ctx_len[] and n_nodes[].
struct CombineArgs {
    const int32_t* ctx_len;
    const int32_t* n_nodes;
    int S, B, H, Hkv, g, nb;
    int G;                    // CTAs of the main kernel
    uint32_t G_magic;         // ceil(2^32 / G)
    int Hw;                   // heads of the work list
    int kv_rows;
    const float* partials;
    __nv_bfloat16* out;
    float* lse;
};

// one round: kCombineRound parts of a row, their (m, l) and 16 columns of O/l, into the running (M, L, acc)
__device__ __forceinline__ void merge_round(const float (&mp)[kCombineRound], const float (&lp)[kCombineRound],
                                            const uint4 (&x)[kCombineRound][2], float& M_run, float& L_run, float (&acc)[16]) {
    float M_new = M_run;
#pragma unroll
    for (int q = 0; q < kCombineRound; ++q) M_new = fmaxf(M_new, mp[q]);
    const float a_old = (M_run == -INFINITY) ? 0.f : ex2(M_run - M_new);
    L_run *= a_old;
#pragma unroll
    for (int u = 0; u < 16; ++u) acc[u] *= a_old;
#pragma unroll
    for (int q = 0; q < kCombineRound; ++q) {
        const float w = ((mp[q] == -INFINITY) ? 0.f : ex2(mp[q] - M_new)) * lp[q];   // un-normalise: O_p = x_p * l_p
        L_run += w;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t hw[4] = {x[q][u].x, x[q][u].y, x[q][u].z, x[q][u].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hw[e]));
                acc[8 * u + 2 * e] += w * f.x;
                acc[8 * u + 2 * e + 1] += w * f.y;
            }
        }
    }
    M_run = M_new;
}
__device__ __forceinline__ void store_merged(__nv_bfloat16* dst, const float (&acc)[16], float L) {
    const float inv = 1.f / L;
#pragma unroll
    for (int u = 0; u < 2; ++u)
        reinterpret_cast<uint4*>(dst)[u] =
            make_uint4(pack_bf16x2(acc[8 * u] * inv, acc[8 * u + 1] * inv), pack_bf16x2(acc[8 * u + 2] * inv, acc[8 * u + 3] * inv),
                       pack_bf16x2(acc[8 * u + 4] * inv, acc[8 * u + 5] * inv), pack_bf16x2(acc[8 * u + 6] * inv, acc[8 * u + 7] * inv));
}

template <bool kGrouped, bool kCounts>
__device__ __forceinline__ void combine_heads(const CombineArgs& ca, int rg, int h, int s) {
    const int32_t* __restrict__ ctx_len = ca.ctx_len;
    const int32_t* __restrict__ n_nodes = kCounts ? ca.n_nodes : nullptr;
    const int S = ca.S, B = ca.B, H = ca.H, G = ca.G;
    const float* __restrict__ partials = ca.partials;
    __nv_bfloat16* __restrict__ out = ca.out;
    float* __restrict__ lse = ca.lse;
    const int Hkv_arg = ca.Hkv, g_arg = ca.g, nb_arg = ca.nb;

    const int Hkv = kGrouped ? Hkv_arg : H, g = kGrouped ? g_arg : 1, nb = kGrouped ? nb_arg : B;
    const int Hw = ca.Hw;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // The partition arithmetic needs only ctx_len[], which is final before this kernel's CTAs can start: the main
    // kernel triggers its dependents after its own pdl_wait(), i.e. after whatever produced ctx_len[] completed.
    // So all of it runs before the wait, and the partial loads are issued the moment the main grid is done.
    Work wk;
    wk.ctx_len = ctx_len; wk.n_nodes = n_nodes; wk.S = S; wk.H = Hw; wk.B = B; wk.G = G; wk.G_magic = ca.G_magic; wk.kv_rows = ca.kv_rows;
    wk.init();
    long long off = 0;
    if (kCounts) for (int ss = 0; ss < s; ++ss) off += (long long)Hw * wk.width(wk.tiles(ss));
    else
#pragma unroll 1
        for (int ss = 0; ss < s; ++ss) off += (long long)Hw * wk.width(wk.tiles(ss));
    const int T = wk.tiles(s);                             // 0: the sequence has no nodes, hence no items and no output
    const long long head_first = off + (long long)h * wk.width(T) + wk.pad;
    const bool any = !kCounts || T > 0;                    // (without counts every sequence has tiles)
    const int c_lo = any ? wk.cta_of(head_first) : 0, c_hi = any ? wk.cta_of(head_first + T - 1) : 0;
    const bool whole = c_lo == c_hi;                       // written directly by the main kernel (or nothing to write)
    const int row = rg * 32 + lane;                        // row of the M tile = (node of the tile, head of the group)
    const int mt = kGrouped ? h / Hkv : 0, hk = h - mt * Hkv;
    const int i_local = kGrouped ? row / g : row, node = mt * nb + i_local;
    const int hq = hk * g + (row - i_local * g);
    const bool row_valid = i_local < nb && node < nodes_of(n_nodes, s, B);
    // CTA c's partial for this head sits in slot 2c, or 2c+1 when its segment starts at the head's first tile,
    // which only the first CTA can do.  With fewer items than CTAs some CTAs in [c_lo, c_hi] are empty.
    const int flag_lo = wk.cta_start<true>(c_lo) <= head_first ? 1 : 0;
    const bool sparse = wk.total < G;
    // every CTA waits, also those with nothing to do: the next kernel in the stream relies on "this grid is
    // complete" implying "the main grid is complete"
    pdl_wait();                                            // the main kernel's partials are complete and visible
    pdl_trigger();
    if (whole || !row_valid) return;
    float M_run = -INFINITY, L_run = 0.f;
    float acc[16];                                         // warp w owns columns 16w .. 16w+15 (column groups 2w, 2w+1)
#pragma unroll
    for (int u = 0; u < 16; ++u) acc[u] = 0.f;

    // kCombineRound parts per round: their (m, l) and their two 16-byte pieces of O/l are loaded together
    // (16 independent loads in flight per thread); a running (M, L) with rescaling merges the rounds
#pragma unroll 1
    for (int cb = c_lo; cb <= c_hi; cb += kCombineRound) {
        float mp[kCombineRound], lp[kCombineRound];
        uint4 x[kCombineRound][2];
#pragma unroll
        for (int q = 0; q < kCombineRound; ++q) {
            const int c = cb + q;
            bool use = c <= c_hi;
            if (use && sparse) use = wk.cta_start<true>(c + 1) > wk.cta_start<true>(c);
            const int sl = use ? 2 * c + (c == c_lo ? flag_lo : 0) : 0;
            const float* pp = partials + (size_t)sl * kUmmaPartFloats;
            mp[q] = use ? __ldcg(pp + kPartHalfWords + row) : -INFINITY;
            lp[q] = use ? __ldcg(pp + kPartHalfWords + kMaxB + row) : 0.f;
            const uint4* p4 = reinterpret_cast<const uint4*>(pp) + row;
#pragma unroll
            for (int u = 0; u < 2; ++u)
                x[q][u] = use ? __ldcg(p4 + (2 * warp + u) * 128) : make_uint4(0u, 0u, 0u, 0u);
        }
        merge_round(mp, lp, x, M_run, L_run, acc);
    }
    store_merged(out + (((size_t)s * B + node) * H + hq) * kHeadDim + 16 * warp, acc, L_run);
    if (lse && warp == 0) lse[((size_t)s * B + node) * H + hq] = (M_run + log2f(L_run)) * kLn2;
}

// the merge as a kernel of its own: grid (row groups of 32, heads of the work list, S)
template <bool kGrouped, bool kCounts>
__global__ void __launch_bounds__(kCombineThreads)
tree_attn_combine_kernel(const CombineArgs ca) {
    combine_heads<kGrouped, kCounts>(ca, blockIdx.x, blockIdx.y, blockIdx.z);
}

// host side: what the merge needs to know about the main kernel's launch (filled by launch_tree_attn_umma)
struct CombinePlan {
    CombineArgs args;
    int row_groups;           // blocks per head
    bool grouped;
    bool valid;               // false: nothing to merge (no tensor-core launch happened)
};

}  // namespace goose
