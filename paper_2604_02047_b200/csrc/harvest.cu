// Harvest of a forward's logits into the Tier-1 (unigram) adjacency table (App. "Aggressive logit harvesting";
// "Dense GPU bigram adjacency table", Tier 1): for every logits row r the k best successor ids and their
// softmax probabilities exp(logit - lse_r) overwrite row row_tok[r] of the two dense [table_rows][k] tensors.
// Rows are harvested in row order, so of several rows that carry the same token the last one wins.  Up to kTableRows rows
// node_topk_kernel writes the table itself.  A call of more rows has this kernel behind it, which decides per row by scanning the later
// rows' tokens (one warp per row on all SMs, no atomics), which keeps the result independent of scheduling.  The top-k and
// the log-sum-exp come from node_topk_kernel.
#include "goose_internal.cuh"

namespace goose {

constexpr int kScatterThreads = 128;

__global__ void __launch_bounds__(kScatterThreads)
harvest_scatter_kernel(const int32_t* __restrict__ row_tok, int rows, int table_rows, int k,
                       const int32_t* __restrict__ ids, const float* __restrict__ vals,
                       const float* __restrict__ row_lse, int32_t* __restrict__ adj_ids,
                       float* __restrict__ adj_scores) {
    const int lane = threadIdx.x & 31;
    const int r = blockIdx.x * (kScatterThreads / 32) + (threadIdx.x >> 5);
    // row_tok[] is an input of the call: the top-k kernel in front lets this one start only after its own wait, so the
    // decision is taken while that kernel still runs (it is a scan of up to `rows` tokens, 47 loads a lane for 1500 rows)
    int tok = -1;
    bool write = false;
    if (r < rows) {
        tok = row_tok[r];
        if (tok >= 0 && tok < table_rows) {                  // else not a table row: skipped
            bool later = false;                              // does a later row carry the same token?
            for (int j = r + 1 + lane; j < rows; j += 32) later |= (row_tok[j] == tok);
            write = !__any_sync(0xFFFFFFFFu, later);
        }
    }
    pdl_wait();
    pdl_trigger();
    if (write && lane < k) {
        adj_ids[(size_t)tok * k + lane] = ids[(size_t)r * k + lane];
        adj_scores[(size_t)tok * k + lane] = expf(vals[(size_t)r * k + lane] - row_lse[r]);
    }
}

cudaError_t launch_harvest_scatter(goose_ctx* c, const HarvestTable& table, int rows, int k, const int32_t* ids, const float* vals,
                                   const float* row_lse, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    dim3 grid((rows + kScatterThreads / 32 - 1) / (kScatterThreads / 32));
    cudaError_t e = launch_pdl(harvest_scatter_kernel, grid, dim3(kScatterThreads), 0, st, table.row_tok, rows,
                               table.table_rows, k, ids, vals, row_lse, table.adj_ids, table.adj_scores);
    c->launches++;
    return e;
}

}  // namespace goose
