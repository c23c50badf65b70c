// Temperature-1 kernels outside the tensor-core engine (Algorithm 1 with
// Decode = a draw from the softmax; verification by lossless speculative
// sampling):
//
// * k_sample_rows — per-(row, column chunk) records of the Gumbel-max keys
//   k = l + g of a logit row (position 0 of the drafting loop draws x_0 from
//   softmax(l_L^(0))).
// * k_lse_rows, k_verify_accept, k_residual_rows, k_residual_merge — speculative
//   sampling
//   (Leviathan et al. 2023; Chen et al. 2023): x_j is accepted when
//   u_j < p_j(x_j) / q_j(x_j); at the first rejection a the bonus token is
//   drawn from max(0, p_a - q_a) (normalised), and after n acceptances from
//   p_n. q_a is rebuilt from the drafting's kept state: the fused row
//   l_L + alpha_a W_vocab r_a - beta_a l_P and its LSE.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "dels_device.cuh"

namespace dels {

namespace {

constexpr int kSampleThreads = 256;

template <typename T>
__device__ __forceinline__ void load8(const T* row, long long c0, long long c1, bool vec, float (&x)[8]);

template <>
__device__ __forceinline__ void load8<uint16_t>(const uint16_t* row, long long c0, long long c1, bool vec,
                                                float (&x)[8]) {
  if (vec && c0 + 8 <= c1) {
    const uint4 w = __ldcs(reinterpret_cast<const uint4*>(row + c0));
    x[0] = bf16lo(w.x); x[1] = bf16hi(w.x); x[2] = bf16lo(w.y); x[3] = bf16hi(w.y);
    x[4] = bf16lo(w.z); x[5] = bf16hi(w.z); x[6] = bf16lo(w.w); x[7] = bf16hi(w.w);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = c0 + i < c1 ? __uint_as_float((uint32_t)row[c0 + i] << 16) : -INFINITY;
  }
}

template <>
__device__ __forceinline__ void load8<float>(const float* row, long long c0, long long c1, bool vec, float (&x)[8]) {
  if (vec && c0 + 8 <= c1) {
    const float4 p = __ldcs(reinterpret_cast<const float4*>(row + c0));
    const float4 q = __ldcs(reinterpret_cast<const float4*>(row + c0 + 4));
    x[0] = p.x; x[1] = p.y; x[2] = p.z; x[3] = p.w;
    x[4] = q.x; x[5] = q.y; x[6] = q.z; x[7] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = c0 + i < c1 ? row[c0 + i] : -INFINITY;
  }
}

// Block-wide merge of the threads' records; thread 0 gets the result.
__device__ __forceinline__ RowAcc block_merge(RowAcc x, RowAcc* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  x = rowacc_warp_reduce(x);
  if (lane == 0) red[warp] = x;
  __syncthreads();
  if (warp == 0) {
    x = lane < (int)(blockDim.x >> 5) ? red[lane] : rowacc_init();
    x = rowacc_warp_reduce(x);
  }
  return x;
}

__device__ __forceinline__ float max8(const float (&x)[8]) {
  return fmaxf(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])), fmaxf(fmaxf(x[4], x[5]), fmaxf(x[6], x[7])));
}

__device__ __forceinline__ float min8(const float (&x)[8]) {
  return fminf(fminf(fminf(x[0], x[1]), fminf(x[2], x[3])), fminf(fminf(x[4], x[5]), fminf(x[6], x[7])));
}

// Top-2 update of eight keys with maximum km: element by element only when
// km exceeds the runner-up (smaller keys change nothing).
__device__ __forceinline__ void push8(const float (&k)[8], float km, int c, float& best, float& second, int& idx) {
  if (km > second) {
#pragma unroll
    for (int i = 0; i < 8; ++i) top2_push(k[i], c + i, best, second, idx);
  }
}

// Records of the keys k_v = l_v + g_v of rows [0, rows): row r is
// src + r * ld; its request index (for the variates) is r / rows_per_request
// and its position j0 + r % rows_per_request. CTA = (row, chunk of
// chunk_cols columns, a multiple of 8). Each thread visits its 8-column
// groups in increasing order (lowest index on exact key ties).
template <typename T>
__global__ void __launch_bounds__(kSampleThreads) k_sample_rows(SampleRowsArgs a) {
  __shared__ RowAcc red[kSampleThreads / 32];
  pdl_wait();
  const int chunk = blockIdx.x % a.nchunks;
  const long long row = blockIdx.x / a.nchunks;
  const int b = (int)(row / a.rows_per_request);
  const int j = a.j0 + (int)(row % a.rows_per_request);
  const T* src = static_cast<const T*>(a.src) + row * a.ld;
  const long long c0 = (long long)chunk * a.chunk_cols;
  const long long c1 = min((long long)a.V, c0 + a.chunk_cols);
  float best = -INFINITY, second = -INFINITY, m = -INFINITY, s = 0.f;
  int idx = 0x7FFFFFFF;
  for (long long c = c0 + 8 * (long long)threadIdx.x; c < c1; c += 8 * kSampleThreads) {
    float x[8], g[8];
    load8<T>(src, c, c1, a.vec != 0, x);
    gumbel8(a.seed, a.step, b, j, a.stream, c >> 3, g);
#pragma unroll
    for (int i = 0; i < 8; ++i) g[i] += x[i];
    push8(g, max8(g), (int)c, best, second, idx);
    lse_chunk_ex2<8>(x, best, m, s);
  }
  RowAcc r;
  r.m = best;
  r.s = s;
  r.second = second;
  r.idx = idx;
  // lse_chunk_ex2 keeps s relative to the running key max: r.m == best
  r = block_merge(r, red);
  if (threadIdx.x == 0)
    reinterpret_cast<float4*>(a.partials)[row * a.partial_ld + chunk] =
        make_float4(r.m, r.s, r.second, __int_as_float(r.idx));
}

// Records (largest value and sum of exponentials) of the target rows, for
// their LSEs: CTA = (row, chunk of chunk_cols columns, a multiple of 8). A
// pure stream of the rows: per element one fused multiply-add, one base-2
// exponential and one addition beside the unpacking, and no top-2 state, which
// the LSE does not need (64 x 17 bf16 rows of 151936: 58 us; the combine's row
// kernel with no short logits and no prior, used before, 81 us).
template <typename T>
__global__ void __launch_bounds__(kSampleThreads, sizeof(T) == 2 ? 6 : 4) k_lse_rows(SampleRowsArgs a) {
  __shared__ RowAcc red[kSampleThreads / 32];
  pdl_wait();
  // not before: launches of this call read weights ahead of their own wait, and
  // the weights may be the work of this launch's predecessor
  if (threadIdx.x == 0) pdl_trigger();
  const int chunk = blockIdx.x % a.nchunks;
  const long long row = blockIdx.x / a.nchunks;
  const long long c0 = (long long)chunk * a.chunk_cols;
  const T* src = static_cast<const T*>(a.src) + row * a.ld + c0;
  const int cols = (int)min((long long)a.chunk_cols, a.V - c0);
  float m = -INFINITY, s = 0.f, nb = 0.f;      // nb = -m log2(e), 0 while m is -inf
  float gate = -INFINITY;                      // m, or -inf while m is past kMaxRef
  // Eight values with maximum vm (NaN ignored). While m is -inf they are -inf
  // (0) or NaN (NaN).
  auto push = [&](float (&x)[8], float vm) {
    if (vm > gate) {
      const float old = m;                     // (-inf: s, 0 or NaN, times 0)
      m = fmaxf(m, vm);
      if (past_ref_bound(m)) {
        s *= ex2_approx((old - m) * kLog2e);
        nb = 0.f;
        gate = -INFINITY;
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] -= m;
      } else {
        nb = -m * kLog2e;
        gate = m;
        s *= ex2_approx(fmaf(old, kLog2e, nb));
      }
    }
    float e[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i & 1] += ex2_approx(fmaf(x[i], kLog2e, nb));
    s += e[0] + e[1];
  };
  if (a.vec) {
    constexpr int W = sizeof(T) == 2 ? 1 : 2;  // 16-byte words per 8 values
    constexpr int U = 4;
    constexpr int step = kSampleThreads * 8;
    // CHECK: the chunk's last, partial block (the others carry no tests)
    auto block = [&](int cb, auto check) {
      constexpr bool CHECK = decltype(check)::value;
      uint4 w[U][W];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (!CHECK || cb + u * step < cols) {
#pragma unroll
          for (int k = 0; k < W; ++k) w[u][k] = __ldcs(reinterpret_cast<const uint4*>(src + cb + u * step) + k);
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (!CHECK || cb + u * step < cols) {
          float x[8];
          if constexpr (W == 1) {
            x[0] = bf16lo(w[u][0].x); x[1] = bf16hi(w[u][0].x); x[2] = bf16lo(w[u][0].y); x[3] = bf16hi(w[u][0].y);
            x[4] = bf16lo(w[u][0].z); x[5] = bf16hi(w[u][0].z); x[6] = bf16lo(w[u][0].w); x[7] = bf16hi(w[u][0].w);
          } else {
#pragma unroll
            for (int k = 0; k < W; ++k) {
              x[4 * k] = __uint_as_float(w[u][k].x); x[4 * k + 1] = __uint_as_float(w[u][k].y);
              x[4 * k + 2] = __uint_as_float(w[u][k].z); x[4 * k + 3] = __uint_as_float(w[u][k].w);
            }
          }
          push(x, max8(x));
        }
    };
    int cb = threadIdx.x * 8;
    const int full = cols / (step * U) * (step * U);
    for (; cb < full; cb += step * U) block(cb, std::false_type{});
    if (cb < cols) block(cb, std::true_type{});
  } else {
    for (int c = threadIdx.x * 8; c < cols; c += 8 * kSampleThreads) {
      float x[8];
      load8<T>(src, c, cols, false, x);
      push(x, max8(x));
    }
  }
  RowAcc r = rowacc_init();
  r.m = m;
  r.s = s;
  r = block_merge(r, red);
  if (threadIdx.x == 0)
    reinterpret_cast<float4*>(a.partials)[row * a.partial_ld + chunk] =
        make_float4(r.m, r.s, r.second, __int_as_float(r.idx));
}

template <typename T>
__device__ __forceinline__ float ld_logit(const void* p, long long i) {
  if constexpr (sizeof(T) == 4) return __ldg(static_cast<const float*>(p) + i);
  else return __uint_as_float((uint32_t)__ldg(static_cast<const uint16_t*>(p) + i) << 16);
}

__device__ __forceinline__ float ld_logit_any(const void* p, int f32, long long i) {
  return f32 ? ld_logit<float>(p, i) : ld_logit<uint16_t>(p, i);
}

// One CTA per request: the LSE of each target row from its records, then the
// acceptance tests, then the gather of the rejected position's
// vocabulary-projection input.
__global__ void __launch_bounds__(256) k_verify_accept(VerifySampledArgs a) {
  __shared__ float lse_s[kMaxSampledBlock + 1];
  __shared__ int acc_s;
  if (threadIdx.x == 0) pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int j = warp; j <= a.n; j += nw) {
    RowAcc x = rowacc_init();
    const long long row = (long long)b * (a.n + 1) + j;
    for (int k = lane; k < a.t_nchunks; k += 32) x = rowacc_merge(x, ld_rowacc_cg(a.t_records, row * a.t_ld + k));
    x = rowacc_warp_reduce(x);
    if (lane == 0) {
      const bool ok = rowacc_valid(x);
      if (!ok) raise_status(a.status, DELS_STATUS_NONFINITE);
      lse_s[j] = ok ? x.m + logf(x.s) : NAN;
    }
  }
  __syncthreads();
  if (warp == 0) {
    // one lane per test (n <= 32), the first that fails ends the block
    bool fails = false, bad = false;
    if (lane < a.n) {
      const int x = a.draft[(long long)b * a.n + lane];
      bad = x < 0 || x >= a.V;
      if (bad) {
        fails = true;
      } else {
        const float t = ld_logit_any(a.target, a.target_f32, ((long long)b * (a.n + 1) + lane) * a.V + x);
        const float ratio = expf((t - lse_s[lane]) - a.draft_lp[(long long)b * a.n + lane]);
        fails = !(uniform_at(a.seed, a.step, b, lane, kStreamAccept, 0) < ratio);
      }
    }
    const unsigned f = __ballot_sync(0xFFFFFFFFu, fails);
    const int acc = f ? __ffs(f) - 1 : a.n;
    if (lane == acc && bad) raise_status(a.status, DELS_STATUS_BAD_TOKEN);
    if (lane == 0) {
      acc_s = acc;
      a.acc[b] = acc;
      a.out_accept[b] = acc;
      a.lse_t[b] = lse_s[acc];
    }
  }
  __syncthreads();
  const int acc = acc_s;
  const int vecs = a.R * a.r_bytes / 16;
  uint4* dst = reinterpret_cast<uint4*>(static_cast<uint8_t*>(a.rg) + (long long)b * a.R * a.r_bytes);
  if (acc >= 1 && acc < a.n && a.state_r) {
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(a.state_r) +
                                                      ((long long)b * a.n + acc) * a.R * a.r_bytes);
    for (int i = threadIdx.x; i < vecs; i += blockDim.x) dst[i] = __ldcg(src + i);
  } else {
    for (int i = threadIdx.x; i < vecs; i += blockDim.x) dst[i] = make_uint4(0, 0, 0, 0);
  }
}

// Eight values of a row for the residual: one or two 16-byte loads (VEC), or
// element by element with -inf past the row's end.
template <typename T, bool VEC>
__device__ __forceinline__ void load8_row(const T* row, int c, int c1, float (&x)[8]) {
  if constexpr (VEC) {
    if constexpr (sizeof(T) == 2) {
      const uint4 w = __ldcs(reinterpret_cast<const uint4*>(row + c));
      x[0] = bf16lo(w.x); x[1] = bf16hi(w.x); x[2] = bf16lo(w.y); x[3] = bf16hi(w.y);
      x[4] = bf16lo(w.z); x[5] = bf16hi(w.z); x[6] = bf16lo(w.w); x[7] = bf16hi(w.w);
    } else {
      const float4 p = __ldcg(reinterpret_cast<const float4*>(row + c));
      const float4 q = __ldcg(reinterpret_cast<const float4*>(row + c) + 1);
      x[0] = p.x; x[1] = p.y; x[2] = p.z; x[3] = p.w;
      x[4] = q.x; x[5] = q.y; x[6] = q.z; x[7] = q.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if constexpr (sizeof(T) == 2) x[i] = c + i < c1 ? bf16_to_f(__ldcg(row + c + i)) : -INFINITY;
      else x[i] = c + i < c1 ? __ldcg(row + c + i) : -INFINITY;
    }
  }
}

// The fast weights flush p and q below 2^-126 to zero, which changes a weight
// p - q noticeably only below 2^-102, so weights up to that are left to a second
// pass with weights of the whole float range. A key of such a weight is at most
// -102 ln 2 - ln(-ln(1 - 2^-24)) = -54.07, so the pass is taken by the threads
// alone whose runner-up ends below that; and p - q <= 2^-102 is not zero only
// for p < 2^-77 (p and q are multiples of 2^-101 above), so only where a target
// logit is that small. (Verification of 64 requests of 151936: 118.4 us without
// the pass, 118.8 with it.)
constexpr float kSmallWeight = 0x1p-102f;
constexpr float kSmallKey = -54.f;

// Records of the bonus draw of request b over one chunk of the vocabulary:
// residual keys log(max(0, p_a - q_a)) + g (a < n) and target keys t + g
// (used after n acceptances, or when every residual weight rounded to zero).
// Issue-bound: the variates and the three transcendentals of the weights are
// most of the instructions. 64 requests of 151936 bf16: 74 us with element
// loads and a top-2 update per element, 42 with 16-byte loads, group tests and
// a grid of one wave (ncu). (Leaving out the groups whose keys, bounded by one
// transform each, lie below a runner-up already met was slower: 54 us.)
template <typename TT, typename TL, bool VEC>
__global__ void __launch_bounds__(kSampleThreads) k_residual_rows(VerifySampledArgs a) {
  __shared__ RowAcc red[kSampleThreads / 32];
  if (threadIdx.x == 0) pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x / a.r_nchunks, chunk = blockIdx.x % a.r_nchunks;
  const int acc = __ldcg(a.acc + b);
  const float lse_t = __ldcg(a.lse_t + b);
  // the rows from this chunk's first column
  const long long c0 = (long long)chunk * a.r_chunk_cols;
  const int cols = (int)min((long long)a.r_chunk_cols, a.V - c0);
  const TT* trow = static_cast<const TT*>(a.target) + ((long long)b * (a.n + 1) + acc) * a.V + c0;
  const bool resid = acc < a.n;
  const TL* lrow = static_cast<const TL*>(a.longp) + ((long long)b * a.n + (resid ? acc : 0)) * a.V + c0;
  const float lse_q = resid ? a.state_lse[(long long)b * a.n + acc] : 0.f;
  const bool head = resid && acc >= 1;
  const float al = head ? a.alpha[acc] : 0.f, nbe = head ? -a.beta[acc] : 0.f;
  const float* ls = a.ls + (long long)b * a.V + c0;
  const float* prior = a.prior ? a.prior + c0 : nullptr;
  float rb = -INFINITY, rs = -INFINITY, pb = -INFINITY, ps = -INFINITY;
  int ri = 0x7FFFFFFF, pi = 0x7FFFFFFF;
  float lo = INFINITY;                      // the smallest target logit met
  auto load_pair = [&](int c, float (&l)[8], float (&sl)[8], float (&pr)[8]) {
    if (resid) load8_row<TL, VEC>(lrow, c, cols, l);
    if (head) {
      load8_row<float, VEC>(ls, c, cols, sl);
      if (prior) load8_row<float, VEC>(prior, c, cols, pr);
    }
  };
  auto fused = [&](float l, float sl, float pr) {
    return head ? fmaf(nbe, prior ? pr : 0.f, fmaf(al, sl, l)) : l;
  };
  auto weight = [&](float t, float x) {
    return ex2_approx((t - lse_t) * kLog2e) - ex2_approx((x - lse_q) * kLog2e);
  };
  for (int c = 8 * (int)threadIdx.x; c < cols; c += 8 * kSampleThreads) {
    float t[8], l[8], sl[8], pr[8];
    load8_row<TT, VEC>(trow, c, cols, t);
    load_pair(c, l, sl, pr);
    float g[8], k[8];
    gumbel8(a.seed, a.step, b, acc, kStreamResidual, (c0 + c) >> 3, g);
#pragma unroll
    for (int i = 0; i < 8; ++i) k[i] = t[i] + g[i];
    push8(k, max8(k), (int)(c0 + c), pb, ps, pi);
    if (resid) {
      lo = fminf(lo, min8(t));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float w = weight(t[i], fused(l[i], sl[i], pr[i]));
        k[i] = w > kSmallWeight && (VEC || c + i < cols) ? fmaf(lg2_approx(w), kLn2, g[i]) : -INFINITY;
      }
      push8(k, max8(k), (int)(c0 + c), rb, rs, ri);
    }
  }
  // the small weights, where they may count (kSmallWeight)
  if (resid && rs < kSmallKey && (lo - lse_t) * kLog2e < -77.f) {
#pragma unroll 1
    for (int c = 8 * (int)threadIdx.x; c < cols; c += 8 * kSampleThreads) {
      float t[8], l[8], sl[8], pr[8];
      load8_row<TT, VEC>(trow, c, cols, t);
      bool small = false;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float p = (t[i] - lse_t) * kLog2e;
        small |= p < -77.f && p > -151.f;
      }
      if (!small) continue;
      load_pair(c, l, sl, pr);
      float g[8], k[8];
      gumbel8(a.seed, a.step, b, acc, kStreamResidual, (c0 + c) >> 3, g);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float x = fused(l[i], sl[i], pr[i]);
        const float w = __expf(t[i] - lse_t) - __expf(x - lse_q);
        k[i] = w > 0.f && !(weight(t[i], x) > kSmallWeight) && (VEC || c + i < cols) ? __logf(w) + g[i] : -INFINITY;
      }
      push8(k, max8(k), (int)(c0 + c), rb, rs, ri);
    }
  }
  RowAcc r;
  r.m = rb; r.s = 1.f; r.second = rs; r.idx = ri;
  RowAcc p;
  p.m = pb; p.s = 1.f; p.second = ps; p.idx = pi;
  r = block_merge(r, red);
  __syncthreads();
  p = block_merge(p, red);
  if (threadIdx.x == 0) {
    float4* out = reinterpret_cast<float4*>(a.r_records) + ((long long)b * a.r_nchunks + chunk) * 2;
    out[0] = make_float4(r.m, r.s, r.second, __int_as_float(r.idx));
    out[1] = make_float4(p.m, p.s, p.second, __int_as_float(p.idx));
  }
}

// One CTA per request: the bonus token from the merged records.
__global__ void __launch_bounds__(256) k_residual_merge(VerifySampledArgs a) {
  __shared__ RowAcc red[8];
  if (threadIdx.x == 0) pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x;
  RowAcc r = rowacc_init(), p = rowacc_init();
  for (int k = threadIdx.x; k < a.r_nchunks; k += blockDim.x) {
    r = rowacc_merge(r, ld_rowacc_cg(a.r_records, ((long long)b * a.r_nchunks + k) * 2));
    p = rowacc_merge(p, ld_rowacc_cg(a.r_records, ((long long)b * a.r_nchunks + k) * 2 + 1));
  }
  r = block_merge(r, red);
  __syncthreads();
  p = block_merge(p, red);
  if (threadIdx.x == 0) {
    const int acc = __ldcg(a.acc + b);
    const bool use_r = acc < a.n && r.m > -INFINITY;
    const RowAcc& x = use_r ? r : p;
    const bool ok = x.m > -INFINITY && x.m < INFINITY;
    if (!ok) raise_status(a.status, DELS_STATUS_NONFINITE);
    a.out_bonus[b] = ok ? x.idx : -1;
    if (a.out_bonus_gap) a.out_bonus_gap[b] = ok ? x.m - x.second : NAN;
  }
}

__global__ void __launch_bounds__(256) k_selftest_gumbel(const uint32_t* __restrict__ bits, float* __restrict__ g,
                                                        long long n) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    g[i] = gumbel_from_bits(bits[i]);
}

}  // namespace

cudaError_t launch_selftest_gumbel(const uint32_t* bits, float* g, long long n, int sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const long long blocks = std::min<long long>((n + 255) / 256, (long long)sms * 8);
  k_selftest_gumbel<<<(unsigned)blocks, 256, 0, s>>>(bits, g, n);
  return cudaGetLastError();
}

cudaError_t launch_verify_accept(const VerifySampledArgs& a, cudaStream_t s) {
  return launch_pdl(k_verify_accept, dim3((unsigned)a.B), dim3(256), 0, s, a);
}

cudaError_t launch_residual_rows(const VerifySampledArgs& a, cudaStream_t s) {
  const dim3 grid((unsigned)(a.B * a.r_nchunks)), block(kSampleThreads);
  using K = void (*)(VerifySampledArgs);
  const K vec[4] = {k_residual_rows<uint16_t, uint16_t, true>, k_residual_rows<uint16_t, float, true>,
                    k_residual_rows<float, uint16_t, true>, k_residual_rows<float, float, true>};
  const K any[4] = {k_residual_rows<uint16_t, uint16_t, false>, k_residual_rows<uint16_t, float, false>,
                    k_residual_rows<float, uint16_t, false>, k_residual_rows<float, float, false>};
  const int k = (a.target_f32 ? 2 : 0) + (a.long_f32 ? 1 : 0);
  return launch_pdl(a.vec ? vec[k] : any[k], grid, block, 0, s, a);
}

cudaError_t launch_residual_merge(const VerifySampledArgs& a, cudaStream_t s) {
  return launch_pdl(k_residual_merge, dim3((unsigned)a.B), dim3(256), 0, s, a);
}

cudaError_t launch_lse_rows(const SampleRowsArgs& a, bool f32, cudaStream_t s) {
  const long long grid = (long long)a.rows * a.nchunks;
  if (grid == 0) return cudaSuccess;
  return f32 ? launch_pdl(k_lse_rows<float>, dim3((unsigned)grid), dim3(kSampleThreads), 0, s, a)
             : launch_pdl(k_lse_rows<uint16_t>, dim3((unsigned)grid), dim3(kSampleThreads), 0, s, a);
}

int lse_slots_per_sm(bool f32) {
  static std::atomic<int> cache[2] = {{-1}, {-1}};   // a property of the kernel, queried once
  if (cache[f32] < 0) {
    int n = 0;
    const cudaError_t e =
        f32 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_lse_rows<float>, kSampleThreads, 0)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_lse_rows<uint16_t>, kSampleThreads, 0);
    cache[f32] = e == cudaSuccess && n > 0 ? n : 0;
  }
  return cache[f32];
}

cudaError_t launch_sample_rows(const SampleRowsArgs& a, bool f32, cudaStream_t s) {
  const long long grid = (long long)a.rows * a.nchunks;
  if (grid == 0) return cudaSuccess;
  return f32 ? launch_pdl(k_sample_rows<float>, dim3((unsigned)grid), dim3(kSampleThreads), 0, s, a)
             : launch_pdl(k_sample_rows<uint16_t>, dim3((unsigned)grid), dim3(kSampleThreads), 0, s, a);
}

}  // namespace dels
