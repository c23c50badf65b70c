// The per-position merge inside a consumer's launch: every CTA that needs the
// next head input merges its requests' records itself (one warp per request)
// and gathers the embedding rows into shared memory, so that the merge costs
// no launch of its own. One CTA per request group writes the decoded outputs.
#pragma once

#include "dels_device.cuh"

namespace dels {

// Tokens of requests b0 .. b0 + nb - 1 (at most one per warp) at position m.j
// into s_tok; the writer's outputs follow the barrier, off the other warps' path.
__device__ __forceinline__ void merge_requests(const MergeArgs& m, int b0, int nb, bool writer, int* s_tok) {
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
  RowAcc x = rowacc_init();
  if (q < nb) {
    const float4* rec = reinterpret_cast<const float4*>(m.partials) + (long long)(b0 + q) * m.partial_ld;
    for (int k = lane; k < m.count; k += 32) x = rowacc_merge(x, ld_rowacc_cg(rec, k));   // mostly one
    __syncwarp();
    x = rowacc_warp_reduce(x);
    if (lane == 0) s_tok[q] = (m.smp.on ? rowacc_valid_sampled(x) : rowacc_valid(x)) ? x.idx : -1;
  }
  __syncthreads();
  if (writer && q < nb && lane == 0)
    decode_record(x, m.smp, b0 + q, m.n, m.j, m.tokens, m.out_lp, m.out_gap, m.status);
}

// 16-byte vector v of request b0 + q's head input (the embedding rows of its
// last m.window tokens, zeros before the block): vecs of them per token row.
__device__ __forceinline__ uint4 gather_vec(const MergeArgs& m, int b0, int q, int v, int vecs, const int* s_tok) {
  const int w = v / vecs, k = v - w * vecs;
  const int j = m.j - w;
  const int tok = w == 0 ? s_tok[q] : j >= 0 ? __ldcg(m.tokens + (long long)(b0 + q) * m.n + j) : -1;
  return tok >= 0 ? __ldg(reinterpret_cast<const uint4*>(m.table) + (long long)tok * vecs + k) : make_uint4(0, 0, 0, 0);
}

}  // namespace dels
