// float32 local heads on CUDA cores: the head products and the vocabulary
// projection fused with the combine.
//
// Both read a weight matrix once for a handful of requests, so they are bound
// by the weights' bytes (L2 for the sizes float32 heads have) as long as
// enough loads are in flight. A warp owns R consecutive weight rows and BG
// requests: each lane takes 4 consecutive k of every 128, so a step is R
// 16-byte weight loads per lane against BG activation vectors in shared
// memory, and the R x BG sums are finished by one transposing reduction
// (R x BG - 1 shuffles instead of 5 per sum), which leaves sum i in lane i.
// Measured on GB300 (ncu, cold caches) against one row per warp with 4-byte
// loads and a shuffle reduction per request, as it was: for 8 requests, the
// vocabulary of 32000 x 256 57 -> 14 us (33 MB of weights: 5 us) and the two
// GRU products of 1536 x 1024 and 1536 x 512 25 + 17 -> 7.3 us in one launch;
// for one request, the vocabulary of 1024 x 128 33 us on 4 CTAs -> 5.3 us on
// 16, where a launch with nothing to do takes about 4. First weights loaded
// before the wait for the predecessor: block of 8 for that request 62 -> 59 us,
// the 8-request block 203 -> 193 us (215 where the vocabulary's chunks are
// several tiles per warp, so those do without).
//
// A launch may let its successor start at once or only after the wait for its
// own predecessor: small calls (one tile per warp) gain from the first (45.4
// us against 47.0), calls that fill the chip from the second, whose waiting
// CTAs otherwise sit beside the running ones (175 -> 161 us for the 8-request
// block).
#include <algorithm>
#include <climits>

#include "merge_rows.cuh"

namespace dels {

namespace {

constexpr int kWarpsF32 = 8;
constexpr int kThreadsF32 = kWarpsF32 * 32;
constexpr size_t kStageLimit = 96 * 1024;    // activations staged in shared memory up to this

template <bool VEC>
__device__ __forceinline__ float4 load4w(const float* p) {
  if constexpr (VEC) return __ldg(reinterpret_cast<const float4*>(p));
  return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}

// The R weight rows from o0 at this lane's k; rows past o_last repeat it (their
// sums are unused).
template <int R, bool VEC>
__device__ __forceinline__ void load_rows(const float* __restrict__ W, int o0, int o_last, int K, int k,
                                          float4 (&w)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r)
    w[r] = k < K ? load4w<VEC>(W + (long long)min(o0 + r, o_last) * K + k) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// acc[r * BG + b] += w[r] . x[b, k .. k + 3]
template <int R, int BG, bool STAGED>
__device__ __forceinline__ void fma_rows(const float4 (&w)[R], const float* x, long long ldx, int nb, int K, int k,
                                         float (&acc)[R * BG]) {
#pragma unroll
  for (int b = 0; b < BG; ++b) {
    float4 v;
    if constexpr (STAGED) v = *reinterpret_cast<const float4*>(x + b * K + k);
    else v = b < nb ? __ldcg(reinterpret_cast<const float4*>(x + b * ldx + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float& s = acc[r * BG + b];
      s = fmaf(w[r].x, v.x, s);
      s = fmaf(w[r].y, v.y, s);
      s = fmaf(w[r].z, v.z, s);
      s = fmaf(w[r].w, v.w, s);
    }
  }
}

// acc[r * BG + b] = sum over this lane's k (k0, k0 + kstep, ..., 4 at a time)
// of W[o0 + r, k] x[b, k]; `w` holds the rows at k0 (load_rows).
// x: [BG][K] in shared memory, or (STAGED false) request rows in global memory.
template <int R, int BG, bool STAGED, bool VEC>
__device__ __forceinline__ void dot_rows(const float* __restrict__ W, int o0, int o_last, int K, const float* x,
                                         long long ldx, int nb, int k0, int kstep, const float4 (&w)[R],
                                         float (&acc)[R * BG]) {
#pragma unroll
  for (int i = 0; i < R * BG; ++i) acc[i] = 0.f;
  if (k0 < K) fma_rows<R, BG, STAGED>(w, x, ldx, nb, K, k0, acc);
#pragma unroll 2
  for (int k = k0 + kstep; k < K; k += kstep) {
    float4 v[R];
    load_rows<R, VEC>(W, o0, o_last, K, k, v);
    fma_rows<R, BG, STAGED>(v, x, ldx, nb, K, k, acc);
  }
}

// Sums v[i] over the warp for every i < NV (a power of two up to 32); lane l
// returns the sum of index l / (32 / NV). Each step halves the values a lane
// carries: it keeps the half its bit selects and receives that half's other sum.
template <int NV>
__device__ __forceinline__ float transpose_reduce(float (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int off = 16;
#pragma unroll
  for (int n = NV; n > 1; n >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) {
      if (i < n / 2) {
        const float send = up ? v[i] : v[i + n / 2];
        const float keep = up ? v[i + n / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, off);
      }
    }
  }
#pragma unroll
  for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], off);
  return v[0];
}

// Requests b0 .. b0 + nb - 1 into shared memory as [BG][K], zeros past nb.
template <int BG>
__device__ __forceinline__ void stage_rows(float* sx, const float* X, long long ldx, int nb, int K) {
  const int nv = K / 4;
  for (int i = threadIdx.x; i < BG * nv; i += kThreadsF32) {
    const int b = i / nv, v = i - b * nv;
    reinterpret_cast<float4*>(sx)[i] = b < nb ? __ldcg(reinterpret_cast<const float4*>(X + b * ldx) + v)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
}

// Y[b, o] = act(sum_k X[b, k] W[o, k]) for up to two independent products with
// the same O (blockIdx.z); blockIdx.x: request group, blockIdx.y: row groups.
// MERGE: the first product's input is the head input of the position that m
// decodes (merge_requests), not X. KS warps split each row group's K (their sums
// are added in order), so that small matrices still fill the chip.
template <int R, int BG, bool STAGED, bool VEC, bool MERGE>
__global__ void __launch_bounds__(kThreadsF32, 2)
    k_gemv_f32(const __grid_constant__ GemvF32Jobs jobs, int B, int O, int act, int ldy, int KS,
               const __grid_constant__ MergeArgs m) {
  extern __shared__ __align__(16) float sx[];
  __shared__ float red[kWarpsF32][32];
  __shared__ int s_tok[MERGE ? BG : 1];
  constexpr int NV = R * BG;
  if (threadIdx.x == 0 && !jobs.late) pdl_trigger();
  const GemvF32Job& jb = jobs.j[blockIdx.z];
  const int b0 = blockIdx.x * BG, nb = min(BG, B - b0);
  const int K = jb.K;
  const float* X = jb.X + (long long)b0 * jb.ldx;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rg = warp / KS, kw = warp % KS;
  const int per = kWarpsF32 / KS * R;
  const int k0 = (kw * 32 + lane) * 4;
  // the first weights go out before the wait: they are not the predecessor's
  float4 w[R];
  load_rows<R, VEC>(jb.W, blockIdx.y * per + rg * R, O - 1, K, k0, w);
  pdl_wait();
  if (threadIdx.x == 0 && jobs.late) pdl_trigger();
  if (MERGE && blockIdx.z == 0) {
    const bool writer = blockIdx.y == 0;
    merge_requests(m, b0, nb, writer, s_tok);
    if (writer)
      for (int q = 0; q < nb; ++q) keep_draft_input(m.smp, b0 + q, m.n, m.j);
    const int vecs = m.D / 4;
    for (int i = threadIdx.x; i < BG * (K / 4); i += kThreadsF32) {
      const int q = i / (K / 4), v = i - q * (K / 4);
      reinterpret_cast<uint4*>(sx)[i] = q < nb ? gather_vec(m, b0, q, v, vecs, s_tok) : make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
  } else if constexpr (STAGED) {
    stage_rows<BG>(sx, X, jb.ldx, nb, K);
  }
  const int idx = lane / (32 / NV), r = idx / BG, b = idx % BG;
  const bool leader = lane % (32 / NV) == 0;
  for (int base = blockIdx.y * per; base < O; base += gridDim.y * per) {
    const int o0 = base + rg * R;
    float acc[NV];
    if (base > (int)(blockIdx.y * per)) load_rows<R, VEC>(jb.W, o0, O - 1, K, k0, w);
    dot_rows<R, BG, STAGED, VEC>(jb.W, o0, O - 1, K, STAGED ? sx : X, jb.ldx, nb, k0, KS * 128, w, acc);
    float s = transpose_reduce<NV>(acc);
    if (KS > 1) {
      red[warp][lane] = s;
      __syncthreads();
      if (kw == 0)
        for (int i = 1; i < KS; ++i) s += red[warp + i][lane];
    }
    if (kw == 0 && leader && b < nb && o0 + r < O) jb.Y[(long long)(b0 + b) * ldy + o0 + r] = act_f(act, s);
    if (KS > 1) __syncthreads();
  }
}

// Vocabulary projection fused with the combine: CTA (chunk, request group)
// computes l_S[v] = W_vocab[v] . feat[b] over its vocabulary chunk, fuses
// l = l_L + alpha l_S - beta l_P (at temperature 1 the top-2 runs over l + g)
// and writes one record per request. ONE: the chunk is one tile per warp, whose
// first weights are loaded before the wait for the predecessor.
template <int R, int BG, bool STAGED, bool ONE>
__global__ void __launch_bounds__(kThreadsF32, 2)
    k_vocab_combine_f32(const __grid_constant__ VocabF32Args a) {
  extern __shared__ __align__(16) float sx[];
  __shared__ RowAcc red[kWarpsF32][32];
  constexpr int NV = R * BG;
  if (threadIdx.x == 0 && ONE) pdl_trigger();
  const int groups = (a.B + BG - 1) / BG;
  const int chunk = blockIdx.x / groups, b0 = (int)(blockIdx.x % groups) * BG;
  const int nb = min(BG, a.B - b0);
  const int v0 = chunk * a.chunk_rows, v1 = min(a.V, v0 + a.chunk_rows);
  const float* X = a.feat + (long long)b0 * a.K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float4 w[R];
  if constexpr (ONE) load_rows<R, true>(a.W, v0 + warp * R, a.V - 1, a.K, lane * 4, w);
  pdl_wait();
  if (threadIdx.x == 0 && !ONE) pdl_trigger();
  if constexpr (STAGED) stage_rows<BG>(sx, X, a.K, nb, a.K);
  const int idx = lane / (32 / NV), r = idx / BG, b = idx % BG;
  const bool mine = lane % (32 / NV) == 0 && b < nb;
  const long long lrow = (long long)(b0 + b) * a.ld_long;
  float best = -INFINITY, second = -INFINITY, m = -INFINITY, s = 0.f;
  int top = INT_MAX;
  for (int o0 = v0 + warp * R; o0 < v1; o0 += kWarpsF32 * R) {
    const int v = o0 + r;
    const bool live = mine && v < v1;
    float l = 0.f, p = 0.f;
    if (live) {
      l = a.long_f32 ? __ldg(static_cast<const float*>(a.longp) + lrow + v)
                     : bf16_to_f(__ldg(static_cast<const uint16_t*>(a.longp) + lrow + v));
      p = __ldg(a.prior + v);
    }
    float acc[NV];
    if constexpr (!ONE) load_rows<R, true>(a.W, o0, a.V - 1, a.K, lane * 4, w);
    dot_rows<R, BG, STAGED, true>(a.W, o0, a.V - 1, a.K, STAGED ? sx : X, a.K, nb, lane * 4, 128, w, acc);
    const float d = transpose_reduce<NV>(acc);
    if (live) {
      const float f[1] = {fmaf(-a.beta, p, fmaf(a.alpha, d, l))};
      const float key = a.smp.on ? f[0] + gumbel_at(a.smp.seed, a.smp.step, b0 + b, a.j, kStreamDraft, v) : f[0];
      top2_push(key, v, best, second, top);
      lse_chunk<1>(f, best, m, s);
    }
  }
  RowAcc x;
  x.m = best; x.s = s; x.second = second; x.idx = top;
  red[warp][lane] = x;
  __syncthreads();
  // request b's lanes of every warp: R rows each
  for (int q = warp; q < nb; q += kWarpsF32) {
    RowAcc y = rowacc_init();
    for (int i = lane; i < kWarpsF32 * R; i += 32) y = rowacc_merge(y, red[i / R][((i % R) * BG + q) * (32 / NV)]);
    y = rowacc_warp_reduce(y);
    if (lane == 0)
      reinterpret_cast<float4*>(a.partials)[(long long)(b0 + q) * a.partial_ld + chunk] =
          make_float4(y.m, y.s, y.second, __int_as_float(y.idx));
  }
}

// Requests per CTA: up to 8 (with 4 rows per warp: 32 sums, one per lane),
// fewer while their activations exceed the staging limit. Where not even one
// request's fit (K > 24576) the activations are read through L2 instead.
int group_size(int B, int K) {
  const int most = B >= 5 ? 8 : B >= 3 ? 4 : B;
  int bg = most;
  while (bg > 0 && (size_t)bg * K * 4 > kStageLimit) bg /= 2;
  return bg > 0 ? bg : most;
}
int rows_per_warp(int bg) { return bg == 8 ? 4 : 8; }
bool staged(int bg, int K) { return (size_t)bg * K * 4 <= kStageLimit; }

template <int R, int BG>
cudaError_t launch_gemv_bg(const GemvF32Jobs& jobs, int B, int O, int act, int ldy, bool stage, bool vec, int KS,
                           dim3 grid, size_t smem, const MergeArgs* merge, cudaStream_t s) {
  auto kern = merge   ? k_gemv_f32<R, BG, true, true, true>
              : stage ? (vec ? k_gemv_f32<R, BG, true, true, false> : k_gemv_f32<R, BG, true, false, false>)
                      : (vec ? k_gemv_f32<R, BG, false, true, false> : k_gemv_f32<R, BG, false, false, false>);
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, grid, dim3(kThreadsF32), smem, s, jobs, B, O, act, ldy, KS, merge ? *merge : MergeArgs{});
}

template <int R, int BG>
cudaError_t launch_vocab_bg(const VocabF32Args& a, bool stage, dim3 grid, size_t smem, cudaStream_t s) {
  const bool one = a.chunk_rows <= kWarpsF32 * R;
  auto kern = stage ? (one ? k_vocab_combine_f32<R, BG, true, true> : k_vocab_combine_f32<R, BG, true, false>)
                    : k_vocab_combine_f32<R, BG, false, false>;
  const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, grid, dim3(kThreadsF32), smem, s, a);
}

}  // namespace

bool gemv_f32_merges(int B, int K) { return staged(group_size(B, K), K); }

cudaError_t launch_gemv_f32(const GemvF32Jobs& jobs, int njobs, int B, int O, int act, int ldy, int sms,
                            cudaStream_t s, const MergeArgs* merge) {
  if (njobs < 1 || njobs > 2 || B < 1 || O < 1) return cudaErrorInvalidValue;
  int K = jobs.j[0].K;
  bool vec = true;
  for (int i = 0; i < njobs; ++i) {
    if (jobs.j[i].K % 4 != 0) return cudaErrorInvalidValue;
    K = std::max(K, jobs.j[i].K);
    vec = vec && (reinterpret_cast<uintptr_t>(jobs.j[i].W) & 15u) == 0;
  }
  const int bg = group_size(B, K), R = rows_per_warp(bg);
  const bool stage = staged(bg, K);
  if (merge && (!stage || !vec)) return cudaErrorInvalidValue;
  const int groups = (B + bg - 1) / bg;
  // K split over the warps of a CTA until about eight warps per SM have work
  // (a split keeps at least one 128-wide step)
  const long long tasks = (long long)((O + R - 1) / R) * groups * njobs;
  int KS = 1;
  while (KS < kWarpsF32 && tasks * KS < 8LL * sms && K >= 256 * KS) KS *= 2;
  const int per = kWarpsF32 / KS * R;
  const int ctas = std::min((O + per - 1) / per, std::max(1, 8 * sms / (groups * njobs)));
  const dim3 grid((unsigned)groups, (unsigned)ctas, (unsigned)njobs);   // ctas: at most 8 per SM
  const size_t smem = stage ? (size_t)bg * K * 4 : 0;
  switch (bg) {
    case 1: return launch_gemv_bg<8, 1>(jobs, B, O, act, ldy, stage, vec, KS, grid, smem, merge, s);
    case 2: return launch_gemv_bg<8, 2>(jobs, B, O, act, ldy, stage, vec, KS, grid, smem, merge, s);
    case 4: return launch_gemv_bg<8, 4>(jobs, B, O, act, ldy, stage, vec, KS, grid, smem, merge, s);
    default: return launch_gemv_bg<4, 8>(jobs, B, O, act, ldy, stage, vec, KS, grid, smem, merge, s);
  }
}

int vocab_f32_chunks(int B, int K, int V, int partial_ld, int sms, int* chunk_rows) {
  const int bg = group_size(B, K), pass = kWarpsF32 * rows_per_warp(bg);
  const int groups = (B + bg - 1) / bg;
  const int most = std::max(1, std::min(partial_ld, 2 * sms / groups));   // one wave of two CTAs per SM
  const int passes = (V + pass - 1) / pass;
  *chunk_rows = (passes + most - 1) / most * pass;
  return (V + *chunk_rows - 1) / *chunk_rows;
}

cudaError_t launch_vocab_combine_f32(const VocabF32Args& a, int nchunks, cudaStream_t s) {
  const int bg = group_size(a.B, a.K);
  const bool stage = staged(bg, a.K);
  const dim3 grid((unsigned)(nchunks * ((a.B + bg - 1) / bg)));
  const size_t smem = stage ? (size_t)bg * a.K * 4 : 0;
  switch (bg) {
    case 1: return launch_vocab_bg<8, 1>(a, stage, grid, smem, s);
    case 2: return launch_vocab_bg<8, 2>(a, stage, grid, smem, s);
    case 4: return launch_vocab_bg<8, 4>(a, stage, grid, smem, s);
    default: return launch_vocab_bg<4, 8>(a, stage, grid, smem, s);
  }
}

}  // namespace dels
