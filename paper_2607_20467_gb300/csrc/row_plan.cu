// The step's row plan, and the choice of its branch in the step graph.  In a file of its own:
// setting a conditional node's value from the device needs relocatable device code.
#include "common.cuh"

namespace dcl {
namespace {

// ------------------------------------------------------------------ step row plan
// One CTA: per sequence the first computed position (0 under full recompute and on a cache
// refresh, the block-aligned prefix end N + Bk*floor((p-N)/Bk) when the stored keys and
// values are that block's, T for a finished row), the row offsets, and the row tables.
__global__ void __launch_bounds__(1024) row_plan_kernel(RowPlan rp, const int32_t* __restrict__ p, int B, int N,
                                                        int T, int Bk, int cached, int update,
                                                        int32_t* __restrict__ x, int window, int mask_id,
                                                        cudaGraphConditionalHandle select,
                                                        const uint16_t* __restrict__ branches) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ int lm_off[];  // [B], then the sequences' first computed positions [B]
  int* st_pos = lm_off + B;
  const int M = T - N;
  if (threadIdx.x == 0) {
    int off = 0, lmoff = 0;
    for (int b = 0; b < B; ++b) {
      const int pb = p[b];
      int start, end = T, cap = T;
      if (pb >= T) {
        start = T;
      } else if (!cached) {
        start = 0;
      } else {
        const int pe = N + Bk * ((pb - N) / Bk);
        start = (rp.pe_cache[b] == pe) ? pe : 0;
        if (update) rp.pe_cache[b] = pe;
        if (cached == 2 && start != 0) {  // dual cache between refreshes: the current block
          end = min(pe + Bk, T);
          cap = end - pb;
        }
      }
      rp.seq_off[b] = off;
      rp.seq_len[b] = end - start;
      rp.kcap[b] = cap;
      st_pos[b] = start;
      off += end - start;
      lm_off[b] = lmoff;
      lmoff += max(end - max(start, N), 0);
    }
    rp.counts[0] = off;
    rp.counts[1] = lmoff;
    if (select) cudaGraphSetConditional(select, branches[(off + 31) >> 5]);
  }
  __syncthreads();
  for (int b = 0; b < B; ++b) {
    const int len = rp.seq_len[b], off = rp.seq_off[b], start = st_pos[b], end = start + len;
    for (int i = threadIdx.x; i < len; i += blockDim.x) {
      rp.row_seq[off + i] = b;
      rp.row_pos[off + i] = start + i;
    }
    if (cached == 2 && window > 0 && p[b] < T) {
      // Eq. remasking over the window positions past the computed rows (the embedding
      // kernel re-masks the computed ones): between refreshes of the dual cache the window
      // runs past the block
      const int pb = p[b], w0 = max(pb, end), w1 = min(pb + window, T);
      for (int t = w0 + threadIdx.x; t < w1; t += blockDim.x) x[(size_t)b * T + t] = mask_id;
    }
    const int s0 = max(start, N);
    for (int i = threadIdx.x; i < end - s0; i += blockDim.x) {
      const int pos = s0 + i;
      rp.lm_src[lm_off[b] + i] = off + (pos - start);
      rp.lm_slot[lm_off[b] + i] = b * M + (pos - N);
    }
  }
}

}  // namespace

cudaError_t row_plan_launch(const RowPlan& rp, const int32_t* p, int batch, int N, int T, int block_len, int cached,
                            int update, int32_t* x, int window, int mask_id,
                            cudaGraphConditionalHandle select, const uint16_t* branches, cudaStream_t stream) {
  if (batch <= 0 || batch > 4096 || (cached && block_len <= 0) || cached < 0 || cached > 2 || (cached == 2 && !x))
    return cudaErrorInvalidValue;
  return launch_pdl(row_plan_kernel, 1, 1024, 2 * sizeof(int) * batch, stream, rp, p, batch, N, T, block_len, cached,
                    update, x, window, mask_id, select, branches);
}

}  // namespace dcl
