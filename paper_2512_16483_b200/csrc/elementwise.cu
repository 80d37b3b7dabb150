// HBM-bound kernels of the path: row score, top-r selection with ballot prefix-sum compaction,
// LayerNorm + AdaLN modulation, restoration fill (bilinear Up of the cached group output), and
// the layout / type conversions between them.  All use 16-byte vector accesses.
#include "internal.h"
#include "ptx.cuh"

namespace fvar {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------------
// Row score s_i = sum_c x[i][c]^2: one warp per row, float4 loads.  Row (e, i) of the compact
// score array reads row xmap(e, i) of x.
// With `noise` (Exp(1) variates, one per row) the value written is the sampling key s_i / E_i: the r
// largest keys are a draw without replacement with probability proportional to s_i.
__global__ void __launch_bounds__(256) row_scores_kernel(const float *__restrict__ x, RowMap xmap, int M,
                                                         long long rows, int C, const float *__restrict__ noise,
                                                         float *__restrict__ scores) {
  pdl_wait();
  pdl_launch_dependents();
  const long long row = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (row >= rows) return;
  const int lane = threadIdx.x & 31;
  const int e = static_cast<int>(row / M), i = static_cast<int>(row - static_cast<long long>(e) * M);
  const float4 *p = reinterpret_cast<const float4 *>(x + (static_cast<long long>(e * xmap.bmul + xmap.boff) * xmap.rpb + i) * C);
  float acc = 0.f;
  for (int c = lane; c < C / 4; c += 32) {
    float4 v = __ldg(p + c);
    acc = fmaf(v.x, v.x, acc);
    acc = fmaf(v.y, v.y, acc);
    acc = fmaf(v.z, v.z, acc);
    acc = fmaf(v.w, v.w, acc);
  }
  acc = warp_sum(acc);
  if (lane == 0) scores[row] = noise ? __fdiv_rn(acc, noise[row]) : acc;
}

cudaError_t launch_row_scores(const float *x, RowMap xmap, int E, int M, int C, const float *noise, float *scores,
                              cudaStream_t st) {
  const long long rows = static_cast<long long>(E) * M;
  if (rows <= 0) return cudaSuccess;
  return launch_pdl(row_scores_kernel, dim3(static_cast<unsigned>((rows + 7) / 8)), dim3(256), 0, st, x, xmap, M, rows, C, noise, scores);
}

// ------------------------------------------------------------------------------------------------
// Top-r selection.  One CTA per batch element.  The fp32 scores map to unsigned keys whose order
// is the float order (NaN -> +inf, -0 -> +0); a 4-pass, 8-bit radix select finds the key of the
// r-th largest; rows are then compacted in ascending index order: every key above the threshold,
// plus the first (r - #above) rows whose key equals it.  Prefix sums use warp ballots.
constexpr int kSelThreads = 1024;

__device__ __forceinline__ unsigned score_key(float s) {
  if (s != s) s = INFINITY;
  s += 0.0f;                                    // -0 -> +0
  const unsigned u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__global__ void __launch_bounds__(kSelThreads) select_topr_kernel(const float *__restrict__ scores, int M, int r,
                                                                  int *__restrict__ idx, int *__restrict__ inv) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ unsigned hist[256];
  __shared__ unsigned s_prefix, s_need;
  __shared__ int warp_gt[32], warp_eq[32];
  __shared__ int base_gt, base_eq;
  const int b = blockIdx.x;
  const float *s = scores + static_cast<long long>(b) * M;
  int *idx_b = idx + static_cast<long long>(b) * r;
  int *inv_b = inv + static_cast<long long>(b) * M;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // radix select: after the loop, `prefix` is the key of the r-th largest and `need` is how many
  // rows with exactly that key are taken
  unsigned prefix = 0, mask = 0, need = static_cast<unsigned>(r);
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    for (int i = tid; i < M; i += kSelThreads) {
      const unsigned k = score_key(s[i]);
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (warp == 0) {
      // Find the digit d at which the count of keys with a larger digit first reaches `need`:
      // lane l owns the 8 bins 255 - 8l ... 248 - 8l; a warp scan gives the count above its range.
      unsigned cnt[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        cnt[j] = hist[255 - 8 * lane - j];
        tot += cnt[j];
      }
      unsigned incl = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      unsigned acc = incl - tot;
      if (acc < need && need <= incl) {          // exactly one lane: the matching set holds >= need keys
        int d = 255 - 8 * lane;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (acc + cnt[j] >= need) break;
          acc += cnt[j];
          --d;
        }
        s_prefix = prefix | (static_cast<unsigned>(d) << shift);
        s_need = need - acc;
      }
    }
    __syncthreads();
    prefix = s_prefix;
    need = s_need;
    mask |= 255u << shift;
    __syncthreads();
  }
  const unsigned thr = prefix;

  if (tid == 0) {
    base_gt = 0;
    base_eq = 0;
  }
  __syncthreads();
  for (int start = 0; start < M; start += kSelThreads) {
    const int i = start + tid;
    const unsigned k = (i < M) ? score_key(s[i]) : 0u;
    const bool gt = (i < M) && k > thr;
    const bool eq = (i < M) && k == thr;
    const unsigned bgt = __ballot_sync(0xffffffffu, gt), beq = __ballot_sync(0xffffffffu, eq);
    if (lane == 0) {
      warp_gt[warp] = __popc(bgt);
      warp_eq[warp] = __popc(beq);
    }
    __syncthreads();
    if (warp == 0) {                           // exclusive scan of the 32 per-warp counts
      int g = warp_gt[lane], q = warp_eq[lane];
      int gi = g, qi = q;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int tg = __shfl_up_sync(0xffffffffu, gi, o), tq = __shfl_up_sync(0xffffffffu, qi, o);
        if (lane >= o) {
          gi += tg;
          qi += tq;
        }
      }
      warp_gt[lane] = gi - g;
      warp_eq[lane] = qi - q;
    }
    __syncthreads();
    const unsigned below = (1u << lane) - 1u;
    const int n_gt = base_gt + warp_gt[warp] + __popc(bgt & below);   // rows above thr before i
    const int n_eq = base_eq + warp_eq[warp] + __popc(beq & below);   // rows equal to thr before i
    if (i < M) {
      const bool take = gt || (eq && n_eq < static_cast<int>(need));
      const int pos = n_gt + min(n_eq, static_cast<int>(need));
      if (take) idx_b[pos] = i;
      inv_b[i] = take ? pos : -1;
    }
    __syncthreads();
    if (tid == kSelThreads - 1) {
      base_gt = n_gt + (gt ? 1 : 0);
      base_eq = n_eq + (eq ? 1 : 0);
    }
    __syncthreads();
  }
}

// The same result for up to 256 rows by counting: row i is taken if fewer than r rows come before it, those with a larger
// key and those with the same key and a lower index.  The M x M comparisons are spread over the block, part p of the rows
// against all of them in warps of their own, so that every read of a key is a broadcast; with k_j >= 1, "k_j >= k_i" for
// j < i and "k_j > k_i" for j > i are one comparison against k_i - 1 and k_i.  No histograms, so three barriers instead of
// two dozen.  Bound by latency; in a chain of itself 169 rows 4.4 -> 3.3 us, 256 rows 4.3 -> 3.7, but 506 rows 4.4 -> 7.2, where the
// comparisons are most of it, hence the line.  In a late step it runs beside the chain, whose QKV product cannot start on
// the SMs that its 1024 threads fill: 13 x 13 scale of the 1024-column stack, eight elements, 1017 -> 1002 us.
constexpr int kSelCountMax = 256;
__global__ void __launch_bounds__(kSelThreads) select_count_kernel(const float *__restrict__ scores, int M, int r,
                                                                   int *__restrict__ idx, int *__restrict__ inv) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ __align__(16) unsigned keys[kSelCountMax];
  __shared__ int before[kSelThreads];
  __shared__ int warp_taken[kSelCountMax / 32];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int width = (M + 31) & ~31, parts = kSelThreads / width, part = tid / width, i = tid - part * width;
  if (tid < kSelCountMax) keys[tid] = tid < M ? score_key(scores[static_cast<long long>(b) * M + tid]) : 0u;    // 0: before nobody
  __syncthreads();
  if (part < parts) {
    const unsigned ki = keys[i];
    const int chunks = (M + 3) / 4, per = (chunks + parts - 1) / parts;
    const int c0 = part * per, c1 = min(chunks, c0 + per), own = i / 4;
    int n = 0;
    auto count = [&](int lo, int hi, unsigned t) {
#pragma unroll 4
      for (int c = lo; c < hi; ++c) {
        const uint4 k = reinterpret_cast<const uint4 *>(keys)[c];
        n += (k.x > t) + (k.y > t) + (k.z > t) + (k.w > t);
      }
    };
    count(c0, min(c1, own), ki - 1u);
    count(max(c0, own + 1), c1, ki);
    if (own >= c0 && own < c1)
#pragma unroll
      for (int e = 0; e < 4; ++e) n += keys[4 * own + e] > (4 * own + e < i ? ki - 1u : ki);
    before[part * width + i] = n;
  }
  __syncthreads();
  bool take = false;
  if (tid < M) {
    int n = 0;
    for (int p = 0; p < parts; ++p) n += before[p * width + tid];
    take = n < r;
  }
  const unsigned taken = __ballot_sync(0xffffffffu, take);
  if (lane == 0 && tid < kSelCountMax) warp_taken[tid >> 5] = __popc(taken);
  __syncthreads();
  if (tid >= M) return;
  int pos = __popc(taken & ((1u << lane) - 1u));
  for (int w = 0; w < tid >> 5; ++w) pos += warp_taken[w];
  if (take) idx[static_cast<long long>(b) * r + pos] = tid;
  inv[static_cast<long long>(b) * M + tid] = take ? pos : -1;
}

cudaError_t launch_select_topr(const float *scores, int B, int M, int r, int *idx, int *inv, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  if (M <= kSelCountMax) return launch_pdl(select_count_kernel, dim3(B), dim3(kSelThreads), 0, st, scores, M, r, idx, inv);
  return launch_pdl(select_topr_kernel, dim3(B), dim3(kSelThreads), 0, st, scores, M, r, idx, inv);
}

// Test hook: take the caller's index lists instead of selecting.  Checks range and strict ascent;
// a bad list sets a status bit and the offending entry is clamped into range.
__global__ void copy_indices_kernel(const int *__restrict__ forced, int M, int r, int ld_forced,
                                    int *__restrict__ idx, int *__restrict__ inv, unsigned *status) {
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.x;
  const int *f = forced + static_cast<long long>(b) * ld_forced;
  int *idx_b = idx + static_cast<long long>(b) * r;
  int *inv_b = inv + static_cast<long long>(b) * M;
  for (int i = threadIdx.x; i < M; i += blockDim.x) inv_b[i] = -1;
  __syncthreads();
  for (int j = threadIdx.x; j < r; j += blockDim.x) {
    int v = f[j];
    const bool bad = v < 0 || v >= M || (j > 0 && f[j - 1] >= v);
    if (bad) atomicOr(status, kStatusBadIndex);
    v = min(max(v, 0), M - 1);
    idx_b[j] = v;
    inv_b[v] = j;
  }
}

cudaError_t launch_copy_indices(const int *forced, int B, int M, int r, int ld_forced, int *idx, int *inv,
                                unsigned *status, cudaStream_t st) {
  return launch_pdl(copy_indices_kernel, dim3(B), dim3(256), 0, st, forced, M, r, ld_forced, idx, inv, status);
}

// ------------------------------------------------------------------------------------------------
// y = LN(x) * (1 + scale) + shift  (or LN(x) * gamma): one CTA of 128 threads per row, the row held in registers as T
// float4 a thread (two-pass mean / variance), bf16 output.
// In the step a row count of 2 .. 8192 is a launch of 1 - 18 us between two GEMMs, so it is the chain of latencies that
// counts: the vectors a row is modulated with are requested together with the row, or before the wait for the preceding
// kernel where the caller says that no kernel in flight writes them (`early`: the step's AdaLN vectors and gamma are
// written by fvar_set_cond only).  Rows x columns, in a chain of such launches, against the form before (warp a row from
// 4096 rows, vectors after the statistics): 16 x 2048 4.8 -> 1.4 us, 400 x 2048 5.6 -> 2.5, 2704 x 1024 5.1 -> 4.7,
// 8192 x 2048 30 -> 18 (5.6 TB/s of 6.5).  Timed one by one inside a step, where no launch overlaps the next, little of
// that is left: 16 x 2048 7.8 before and after, a launch of three dense d16 scales 11.4 -> 10.6, of three dense Infinity
// scales 22.2 -> 20.9; one that adds K ranges up takes longer (three late Infinity scales 8.1 -> 8.5).  A warp or two a
// row, or two rows a CTA, are level at best.
constexpr int kLnThreads = 128;
constexpr int kLnMaxVec = 16;                   // float4 a thread: 8192 columns

// PARTS: the row is completed first, x += gate * (sum of the K ranges of the GEMM before it, in range order, + bias),
// and written back; the reads of the ranges hide in the latency that the row's own have.
template <int T, bool PARTS>
__global__ void __launch_bounds__(kLnThreads) ln_modulate_kernel(const float *x, RowMap xmap, int rows, int C,
                                                                 const float *__restrict__ shift, const float *__restrict__ scale,
                                                                 long long vec_stride, int bmul, int boff, const bf16 *__restrict__ gamma,
                                                                 float eps, int early, bf16 *__restrict__ y, GemmParts parts) {
  pdl_launch_dependents();      // nothing precedes the wait but loads: the successor may start its own prologue right away
  __shared__ float red[2][kLnThreads / 32];
  constexpr bool kHold = T <= 4;                // the vectors fit in registers beside the row
  const int e = blockIdx.x / rows, j = blockIdx.x - e * rows;
  const int n4 = C / 4, tid = threadIdx.x;
  const long long voff = static_cast<long long>(e * bmul + boff) * vec_stride;
  float4 mul[kHold ? T : 1], add[kHold ? T : 1];
  auto vec_mul = [&](int g) {                   // what the normalised value is multiplied with ...
    if (gamma == nullptr) {
      const float4 s = __ldg(reinterpret_cast<const float4 *>(scale + voff) + g);
      return make_float4(1.0f + s.x, 1.0f + s.y, 1.0f + s.z, 1.0f + s.w);
    }
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(gamma) + g);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
  };
  auto vec_add = [&](int g) {                   // ... and what is added
    return gamma == nullptr ? __ldg(reinterpret_cast<const float4 *>(shift + voff) + g) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto fetch_vecs = [&]() {
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (tid + t * kLnThreads < n4) { mul[kHold ? t : 0] = vec_mul(tid + t * kLnThreads); add[kHold ? t : 0] = vec_add(tid + t * kLnThreads); }
  };
  if (kHold && early) fetch_vecs();
  float4 gate[PARTS ? T : 1], bias[PARTS ? T : 1];
  if constexpr (PARTS) {
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const int g = tid + t * kLnThreads;
      if (g >= n4) continue;
      gate[t] = __ldg(reinterpret_cast<const float4 *>(parts.gate + voff) + g);
      const uint2 u = parts.bias ? __ldg(reinterpret_cast<const uint2 *>(parts.bias) + g) : make_uint2(0u, 0u);
      const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
      bias[t] = make_float4(a.x, a.y, b.x, b.y);
    }
  }
  pdl_wait();
  if (kHold && !early) fetch_vecs();
  const RowMap rmap = PARTS ? parts.inmap : xmap;
  const float4 *xr = reinterpret_cast<const float4 *>((PARTS ? parts.xin : x) + (static_cast<long long>(e * rmap.bmul + rmap.boff) * rmap.rpb + j) * C);
  float4 v[T];
  float sum = 0.f;
#pragma unroll
  for (int t = 0; t < T; ++t) v[t] = tid + t * kLnThreads < n4 ? xr[tid + t * kLnThreads] : make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (PARTS) {
    const float4 *pr = reinterpret_cast<const float4 *>(parts.part + static_cast<long long>(blockIdx.x) * C);
    float4 *xw = reinterpret_cast<float4 *>(const_cast<float *>(x) + (static_cast<long long>(e * xmap.bmul + xmap.boff) * xmap.rpb + j) * C);
    float4 q[kMaxParts][T];
#pragma unroll
    for (int s = 0; s < kMaxParts; ++s)
#pragma unroll
      for (int t = 0; t < T; ++t)
        q[s][t] = (s < parts.splits && tid + t * kLnThreads < n4) ? pr[s * (parts.stride >> 2) + tid + t * kLnThreads] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      if (tid + t * kLnThreads >= n4) continue;
      float4 a = q[0][t];
#pragma unroll
      for (int s = 1; s < kMaxParts; ++s) { a.x += q[s][t].x; a.y += q[s][t].y; a.z += q[s][t].z; a.w += q[s][t].w; }
      a.x += bias[t].x; a.y += bias[t].y; a.z += bias[t].z; a.w += bias[t].w;
      v[t].x = fmaf(gate[t].x, a.x, v[t].x); v[t].y = fmaf(gate[t].y, a.y, v[t].y);
      v[t].z = fmaf(gate[t].z, a.z, v[t].z); v[t].w = fmaf(gate[t].w, a.w, v[t].w);
      xw[tid + t * kLnThreads] = v[t];
    }
  }
#pragma unroll
  for (int t = 0; t < T; ++t) sum += (v[t].x + v[t].y) + (v[t].z + v[t].w);
  auto block_sum = [&](float val, int k) {
    val = warp_sum(val);
    if ((tid & 31) == 0) red[k][tid >> 5] = val;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kLnThreads / 32; ++w) tot += red[k][w];
    return tot;
  };
  const float mean = block_sum(sum, 0) / C;
  float sq = 0.f;
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (tid + t * kLnThreads < n4) {
      const float a = v[t].x - mean, b = v[t].y - mean, c = v[t].z - mean, d = v[t].w - mean;
      sq = fmaf(a, a, sq); sq = fmaf(b, b, sq); sq = fmaf(c, c, sq); sq = fmaf(d, d, sq);
    }
  const float rstd = rsqrtf(block_sum(sq, 1) / C + eps);
  uint2 *yr = reinterpret_cast<uint2 *>(y + static_cast<long long>(blockIdx.x) * C);
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int g = tid + t * kLnThreads;
    if (g < n4) {
      const float4 m = kHold ? mul[kHold ? t : 0] : vec_mul(g), h = kHold ? add[kHold ? t : 0] : vec_add(g);
      const __nv_bfloat162 o0 = __floats2bfloat162_rn(fmaf((v[t].x - mean) * rstd, m.x, h.x), fmaf((v[t].y - mean) * rstd, m.y, h.y));
      const __nv_bfloat162 o1 = __floats2bfloat162_rn(fmaf((v[t].z - mean) * rstd, m.z, h.z), fmaf((v[t].w - mean) * rstd, m.w, h.w));
      yr[g] = make_uint2(*reinterpret_cast<const uint32_t *>(&o0), *reinterpret_cast<const uint32_t *>(&o1));
    }
  }
}

cudaError_t launch_ln_modulate(const float *x, RowMap xmap, int E, int rows, int C, const float *shift,
                               const float *scale, long long vec_stride, int bmul, int boff, const bf16 *gamma,
                               float eps, bool early, bf16 *y, cudaStream_t st) {
  if (E * rows <= 0) return cudaSuccess;
  if (C % 8 != 0 || C > 4 * kLnThreads * kLnMaxVec) return cudaErrorInvalidValue;
  auto go = [&](auto kern) {
    return launch_pdl(kern, dim3(E * rows), dim3(kLnThreads), 0, st, x, xmap, rows, C, shift, scale, vec_stride, bmul, boff, gamma, eps, early ? 1 : 0, y, GemmParts{});
  };
  if (C <= 512) return go(ln_modulate_kernel<1, false>);
  if (C <= 1024) return go(ln_modulate_kernel<2, false>);
  if (C <= 2048) return go(ln_modulate_kernel<4, false>);
  if (C <= 4096) return go(ln_modulate_kernel<8, false>);
  return go(ln_modulate_kernel<16, false>);
}

// C <= 2048: gemm_partial_plan takes no wider output.  (512 columns and fewer have too few tiles for K ranges on a B200, so they have no
// variant of their own.)
cudaError_t launch_ln_parts(float *x, RowMap xmap, int E, int rows, int C, const GemmParts &parts, const float *shift, const float *scale,
                            long long vec_stride, int bmul, int boff, float eps, bf16 *y, cudaStream_t st) {
  if (E * rows <= 0) return cudaSuccess;
  if (C % 8 != 0 || C > 2048 || parts.splits < 1 || parts.splits > kMaxParts || parts.stride % 4 != 0) return cudaErrorInvalidValue;
  auto go = [&](auto kern) {
    return launch_pdl(kern, dim3(E * rows), dim3(kLnThreads), 0, st, static_cast<const float *>(x), xmap, rows, C, shift, scale, vec_stride, bmul, boff,
                      static_cast<const bf16 *>(nullptr), eps, 1, y, parts);
  };
  if (C <= 1024) return go(ln_modulate_kernel<2, true>);
  return go(ln_modulate_kernel<4, true>);
}

// The K ranges of a group's last fc2 (see launch_finish_parts): one CTA of 128 threads a row, T float4 a thread, everything a
// row reads in flight together.  Bound by latency and by the 4 C (ranges + 2) bytes a row, or 4 C more with the split, that
// come from and stay in L2: in the chain about 3 us for 400 rows of 2048 columns in four ranges.  gemm_partial_plan has what the
// GEMM and this launch take together against a GEMM that reduces by itself.
template <int T>
__global__ void __launch_bounds__(kLnThreads) finish_parts_kernel(GemmParts parts, int rows, int C, long long vec_stride, int bmul, int boff,
                                                                  float *out, RowMap omap, const int *__restrict__ scatter,
                                                                  bf16 *__restrict__ xsplit, int xsplit_mk) {
  const int e = blockIdx.x / rows, j = blockIdx.x - e * rows, n4 = C / 4, tid = threadIdx.x;
  float4 gate[T];
  uint2 bias[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int g = tid + t * kLnThreads;
    if (g >= n4) continue;
    gate[t] = __ldg(reinterpret_cast<const float4 *>(parts.gate + static_cast<long long>(e * bmul + boff) * vec_stride) + g);
    bias[t] = parts.bias ? __ldg(reinterpret_cast<const uint2 *>(parts.bias) + g) : make_uint2(0u, 0u);
  }
  pdl_wait();
  pdl_launch_dependents();
  const int jo = scatter ? scatter[static_cast<long long>(e) * rows + j] : j;
  const float4 *xr = reinterpret_cast<const float4 *>(parts.xin + (static_cast<long long>(e * parts.inmap.bmul + parts.inmap.boff) * parts.inmap.rpb + j) * C);
  const float4 *pr = reinterpret_cast<const float4 *>(parts.part + static_cast<long long>(blockIdx.x) * C);
  float4 v[T], q[kMaxParts][T];
#pragma unroll
  for (int t = 0; t < T; ++t)
    if (tid + t * kLnThreads < n4) v[t] = xr[tid + t * kLnThreads];
#pragma unroll
  for (int s = 0; s < kMaxParts; ++s)
#pragma unroll
    for (int t = 0; t < T; ++t)
      q[s][t] = (s < parts.splits && tid + t * kLnThreads < n4) ? pr[s * (parts.stride >> 2) + tid + t * kLnThreads] : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 *dst = reinterpret_cast<float4 *>(out + (static_cast<long long>(e * omap.bmul + omap.boff) * omap.rpb + jo) * C);
  uint2 *hi = xsplit ? reinterpret_cast<uint2 *>(xsplit + (static_cast<long long>(e) * 2 * xsplit_mk + jo) * C) : nullptr;
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int g = tid + t * kLnThreads;
    if (g >= n4) continue;
    float4 a = q[0][t];
#pragma unroll
    for (int s = 1; s < kMaxParts; ++s) { a.x += q[s][t].x; a.y += q[s][t].y; a.z += q[s][t].z; a.w += q[s][t].w; }
    const float2 b0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&bias[t].x)), b1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&bias[t].y));
    a.x = fmaf(gate[t].x, a.x + b0.x, v[t].x); a.y = fmaf(gate[t].y, a.y + b0.y, v[t].y);
    a.z = fmaf(gate[t].z, a.z + b1.x, v[t].z); a.w = fmaf(gate[t].w, a.w + b1.y, v[t].w);
    dst[g] = a;
    if (hi != nullptr) {
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
      const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
      const __nv_bfloat162 l0 = __floats2bfloat162_rn(a.x - f0.x, a.y - f0.y), l1 = __floats2bfloat162_rn(a.z - f1.x, a.w - f1.y);
      hi[g] = make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
      hi[static_cast<long long>(xsplit_mk) * n4 + g] = make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
    }
  }
}

cudaError_t launch_finish_parts(const GemmParts &parts, int E, int rows, int C, long long vec_stride, int bmul, int boff, float *out, RowMap omap,
                                const int *scatter, bf16 *xsplit, int xsplit_mk, cudaStream_t st) {
  if (E * rows <= 0) return cudaSuccess;
  if (C % 8 != 0 || C > 2048 || parts.splits < 1 || parts.splits > kMaxParts || parts.stride % 4 != 0) return cudaErrorInvalidValue;
  auto go = [&](auto kern) {
    return launch_pdl(kern, dim3(E * rows), dim3(kLnThreads), 0, st, parts, rows, C, vec_stride, bmul, boff, out, omap, scatter, xsplit, xsplit_mk);
  };
  if (C <= 1024) return go(finish_parts_kernel<2>);
  return go(finish_parts_kernel<4>);
}

// ------------------------------------------------------------------------------------------------
// Restoration fill: rows outside the index set take the bilinearly upsampled cached row
// (half-pixel centres, source coordinate clamped at 0, neighbours clamped at the edge).
// One warp per output row; rows inside the index set are skipped.  Bound by latency and by the map's way to
// memory.  In a late step it runs beside the QKV product, whose blocks leave 11 K registers of an SM: four rows a block of at most 64
// registers a thread fit beside it (8 bytes spill), eight of 56 waited for it to end and then held the SMs that the attention needs
// whole: a step of 404 rows of 1920 columns 2393 -> 2301 us, of 2048 rows 7320 -> 7238, of 1616 or 680 rows of 1024 columns level.  At 40
// registers 128 bytes spill: 2360, 7477.  By itself 5.2 -> 4.8 us for 16 x 128 rows of 1024 columns.
constexpr int kFillThreads = 128;
__global__ void __launch_bounds__(kFillThreads, 8) rtr_fill_kernel(const float *__restrict__ prev, float *__restrict__ out, int E,
                                                       int bmul, int boff, int h0, int w0, int h1, int w1, int C,
                                                       const int *__restrict__ inv, bf16 *__restrict__ xsplit, int mk) {
  pdl_wait();
  pdl_launch_dependents();
  const int M1 = h1 * w1;
  const long long gw = static_cast<long long>(blockIdx.x) * (kFillThreads / 32) + (threadIdx.x >> 5);
  if (gw >= static_cast<long long>(E) * M1) return;
  const int e = static_cast<int>(gw / M1), i = static_cast<int>(gw - static_cast<long long>(e) * M1);
  if (inv != nullptr && inv[static_cast<long long>(e) * M1 + i] >= 0) return;
  const int b = e * bmul + boff;
  const int y = i / w1, xq = i - y * w1;
  const BilinearTap tap = bilinear_tap(y, xq, h0, w0, h1, w1);
  const int y0 = tap.y0, y1 = tap.y1, x0 = tap.x0, x1 = tap.x1;
  const float *src = prev + static_cast<long long>(b) * h0 * w0 * C;
  const float4 *p00 = reinterpret_cast<const float4 *>(src + (static_cast<long long>(y0) * w0 + x0) * C);
  const float4 *p01 = reinterpret_cast<const float4 *>(src + (static_cast<long long>(y0) * w0 + x1) * C);
  const float4 *p10 = reinterpret_cast<const float4 *>(src + (static_cast<long long>(y1) * w0 + x0) * C);
  const float4 *p11 = reinterpret_cast<const float4 *>(src + (static_cast<long long>(y1) * w0 + x1) * C);
  float4 *dst = reinterpret_cast<float4 *>(out + (static_cast<long long>(b) * M1 + i) * C);
  uint2 *hi_dst = xsplit ? reinterpret_cast<uint2 *>(xsplit + (static_cast<long long>(e) * 2 * mk + i) * C) : nullptr;
  const long long lo_off = static_cast<long long>(mk) * C / 4;      // in 4-element groups
  const float w00 = tap.w00, w01 = tap.w01, w10 = tap.w10, w11 = tap.w11;
#pragma unroll 4
  for (int c = threadIdx.x & 31; c < C / 4; c += 32) {
    const float4 a = __ldg(p00 + c), bq = __ldg(p01 + c), cq = __ldg(p10 + c), d = __ldg(p11 + c);
    float4 o;
    o.x = w00 * a.x + w01 * bq.x + w10 * cq.x + w11 * d.x;
    o.y = w00 * a.y + w01 * bq.y + w10 * cq.y + w11 * d.y;
    o.z = w00 * a.z + w01 * bq.z + w10 * cq.z + w11 * d.z;
    o.w = w00 * a.w + w01 * bq.w + w10 * cq.w + w11 * d.w;
    __stcs(dst + c, o);                          // written once, read by a later kernel: stream it
    if (hi_dst != nullptr) {
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(o.x, o.y), h1 = __floats2bfloat162_rn(o.z, o.w);
      const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
      const __nv_bfloat162 l0 = __floats2bfloat162_rn(o.x - f0.x, o.y - f0.y), l1 = __floats2bfloat162_rn(o.z - f1.x, o.w - f1.y);
      hi_dst[c] = make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
      hi_dst[lo_off + c] = make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
    }
  }
}

cudaError_t launch_rtr_fill(const float *prev, float *out, int E, int bmul, int boff, int h0, int w0, int h1, int w1,
                            int C, const int *inv, bf16 *xsplit, int mk, cudaStream_t st) {
  const long long warps = static_cast<long long>(E) * h1 * w1;
  if (warps <= 0) return cudaSuccess;
  return launch_pdl(rtr_fill_kernel, dim3(static_cast<unsigned>((warps + kFillThreads / 32 - 1) / (kFillThreads / 32))), dim3(kFillThreads), 0, st, prev, out, E, bmul, boff, h0, w0, h1, w1, C,
                                                                         inv, xsplit, mk);
}

// ------------------------------------------------------------------------------------------------
// Projection drawn from a seed (Q_ij ~ N(0, 1/r), Sec. 3.3 RP of the paper).  Philox4x32-10 (Salmon et
// al., SC'11): call t, counter (t, group, scale, 0) under key (seed low, seed high), gives elements
// 4t .. 4t + 3 of Q^T flattened row-major (element n = j * M + i is Q_ij).  Uniforms u = (x + 0.5) 2^-32,
// Box-Muller on the word pairs (0, 1) and (2, 3) in fp64, one rounding to bf16.  Each value is written
// to both halves of the stored [Q^T | Q^T] row (row stride 2 * Mk).
__device__ __forceinline__ void philox_round(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
  const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
  const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
  const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
  c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
}

__global__ void __launch_bounds__(256) generate_projection_kernel(bf16 *__restrict__ qt, int M, int Mk, int r,
                                                                  uint32_t key0, uint32_t key1, uint32_t group,
                                                                  uint32_t scale) {
  const long long n_total = static_cast<long long>(M) * r;
  const long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (4 * t >= n_total) return;
  uint32_t c[4] = {static_cast<uint32_t>(t), group, scale, 0u};
  uint32_t k0 = key0, k1 = key1;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    philox_round(c, k0, k1);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  const double sqrt_r = sqrt(static_cast<double>(r));
  double z[4];
#pragma unroll
  for (int a = 0; a < 4; a += 2) {
    const double u0 = (static_cast<double>(c[a]) + 0.5) * 0x1p-32, u1 = (static_cast<double>(c[a + 1]) + 0.5) * 0x1p-32;
    const double rad = sqrt(-2.0 * log(u0)), ang = (2.0 * 3.141592653589793) * u1;
    z[a] = rad * cos(ang);
    z[a + 1] = rad * sin(ang);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long n = 4 * t + q;
    if (n < n_total) {
      const int j = static_cast<int>(n / M), i = static_cast<int>(n - static_cast<long long>(j) * M);
      const bf16 v = __double2bfloat16(z[q] / sqrt_r);
      qt[static_cast<long long>(j) * 2 * Mk + i] = v;
      qt[static_cast<long long>(j) * 2 * Mk + Mk + i] = v;
    }
  }
}

cudaError_t launch_generate_projection(bf16 *qt, int M, int Mk, int r, unsigned long long seed, int group, int scale,
                                       cudaStream_t st) {
  const long long calls = (static_cast<long long>(M) * r + 3) / 4;
  if (calls <= 0) return cudaSuccess;
  generate_projection_kernel<<<static_cast<unsigned>((calls + 255) / 256), 256, 0, st>>>(
      qt, M, Mk, r, static_cast<uint32_t>(seed & 0xFFFFFFFFull), static_cast<uint32_t>(seed >> 32),
      static_cast<uint32_t>(group), static_cast<uint32_t>(scale));
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// bf16 tokens -> the fp32 work stream, for the E batch elements the step computes only: computed element e is read
// at element e * smul + soff of `tok` and written at element e * bmul + boff of `x`.
__global__ void tokens_to_f32_kernel(const bf16 *__restrict__ tok, float *__restrict__ x, long long n8, long long per8,
                                     bf16 *__restrict__ xsplit, long long half8, int smul, int soff, int bmul, int boff) {
  pdl_wait();
  pdl_launch_dependents();
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n8) return;
  const long long e = i / per8, off = i - e * per8;
  const uint4 u = __ldg(reinterpret_cast<const uint4 *>(tok) + (e * smul + soff) * per8 + off);
  if (xsplit != nullptr) {                       // hi = the token itself, lo = 0
    uint4 *dst = reinterpret_cast<uint4 *>(xsplit) + e * 2 * half8 + off;
    dst[0] = u;
    dst[half8] = make_uint4(0u, 0u, 0u, 0u);
  }
  const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
  const float2 a = __bfloat1622float2(h[0]), b = __bfloat1622float2(h[1]), c = __bfloat1622float2(h[2]),
               d = __bfloat1622float2(h[3]);
  float4 *dst = reinterpret_cast<float4 *>(x) + 2 * ((e * bmul + boff) * per8 + off);
  dst[0] = make_float4(a.x, a.y, b.x, b.y);
  dst[1] = make_float4(c.x, c.y, d.x, d.y);
}

cudaError_t launch_tokens_to_f32(const bf16 *tok, float *x, int E, int M, int C, bf16 *xsplit, int mk, int smul, int soff,
                                 int bmul, int boff, cudaStream_t st) {
  const long long per8 = static_cast<long long>(M) * C / 8, n8 = static_cast<long long>(E) * per8;
  if (n8 <= 0) return cudaSuccess;
  return launch_pdl(tokens_to_f32_kernel, dim3(static_cast<unsigned>((n8 + 255) / 256)), dim3(256), 0, st, tok, x, n8, per8, xsplit,
                    static_cast<long long>(mk) * C / 8, smul, soff, bmul, boff);
}

__global__ void out_to_bf16_kernel(const float *__restrict__ x, RowMap xmap, int M, int C, bf16 *__restrict__ out) {
  pdl_wait();
  pdl_launch_dependents();
  const int e = blockIdx.y;
  const long long per = static_cast<long long>(M) * C / 8;
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= per) return;
  const float4 *src = reinterpret_cast<const float4 *>(x + static_cast<long long>(e * xmap.bmul + xmap.boff) * xmap.rpb * C);
  const float4 a = src[2 * i], b = src[2 * i + 1];
  __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w),
                 h2 = __floats2bfloat162_rn(b.x, b.y), h3 = __floats2bfloat162_rn(b.z, b.w);
  uint4 u = make_uint4(*reinterpret_cast<uint32_t *>(&h0), *reinterpret_cast<uint32_t *>(&h1),
                       *reinterpret_cast<uint32_t *>(&h2), *reinterpret_cast<uint32_t *>(&h3));
  reinterpret_cast<uint4 *>(out + static_cast<long long>(e) * M * C)[i] = u;
}

cudaError_t launch_out_to_bf16(const float *x, RowMap xmap, int E, int M, int C, bf16 *out, cudaStream_t st) {
  const long long per = static_cast<long long>(M) * C / 8;
  dim3 grid(static_cast<unsigned>((per + 255) / 256), E);
  return launch_pdl(out_to_bf16_kernel, dim3(grid), dim3(256), 0, st, x, xmap, M, C, out);
}

__global__ void silu_bf16_kernel(const bf16 *__restrict__ in, bf16 *__restrict__ out, long long n) {
  pdl_wait();
  pdl_launch_dependents();
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float v = __bfloat162float(in[i]);
  out[i] = __float2bfloat16_rn(v / (1.0f + __expf(-v)));
}

cudaError_t launch_silu_bf16(const bf16 *in, bf16 *out, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  return launch_pdl(silu_bf16_kernel, dim3(static_cast<unsigned>((n + 255) / 256)), dim3(256), 0, st, in, out, n);
}

// Self-test of the bounded wait every kernel of the library relies on: one thread initialises an mbarrier that
// nothing will ever signal and waits on it with the given budget.  The wait gives up, flags the status word
// (kStatusTimeout) and the kernel returns normally: no trap, no fault, the context stays usable.
__global__ void wait_selftest_kernel(long long cycles, unsigned *status) {
  __shared__ unsigned long long bar;
  __shared__ volatile int abort_flag;
  pdl_wait();
  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    mbar_fence_init();
    mbar_wait(smem_u32(&bar), 0, status, &abort_flag, wait_budget(cycles));
  }
}

cudaError_t launch_wait_selftest(long long cycles, unsigned *status, cudaStream_t st) {
  return launch_pdl(wait_selftest_kernel, dim3(1), dim3(32), 0, st, cycles, status);
}

// Asks L2 to fetch [ptr, ptr + bytes): one bulk prefetch of up to 16 KiB per thread.  The range must hold data that no
// kernel in flight writes (weights), so the requests go out before the wait that keeps stream order transitive.
__global__ void l2_prefetch_kernel(const uint8_t *__restrict__ ptr, unsigned long long bytes) {
  pdl_launch_dependents();
  const unsigned long long o = (static_cast<unsigned long long>(blockIdx.x) * blockDim.x + threadIdx.x) * 16384ull;
  if (o < bytes) {
    const unsigned long long n = bytes - o < 16384ull ? bytes - o : 16384ull;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(ptr + o), "r"(static_cast<uint32_t>(n)) : "memory");
  }
  pdl_wait();
}

cudaError_t launch_l2_prefetch(const void *ptr, unsigned long long bytes, cudaStream_t st) {
  bytes &= ~15ull;
  if (bytes == 0) return cudaSuccess;
  const unsigned long long pieces = (bytes + 16383ull) / 16384ull;
  return launch_pdl(l2_prefetch_kernel, dim3(static_cast<unsigned>((pieces + 31) / 32)), dim3(32), 0, st,
                    static_cast<const uint8_t *>(ptr), bytes);
}

// K, V [B][L][H*D] -> cache layout K [B][H][L_cap][D], V^T [B][H][D][L_cap] (one block's worth).
__global__ void load_kv_kernel(const bf16 *__restrict__ K, const bf16 *__restrict__ V, int L, int H, int D, int L_cap,
                               bf16 *__restrict__ kc, bf16 *__restrict__ vt) {
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.z, h = blockIdx.y;
  const int C = H * D;
  for (long long t = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; t < static_cast<long long>(L) * D;
       t += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int l = static_cast<int>(t / D), d = static_cast<int>(t - static_cast<long long>(l) * D);
    const long long src = (static_cast<long long>(b) * L + l) * C + h * D + d;
    kc[((static_cast<long long>(b) * H + h) * L_cap + l) * D + d] = K[src];
    vt[((static_cast<long long>(b) * H + h) * D + d) * L_cap + l] = V[src];
  }
}

cudaError_t launch_load_kv(const bf16 *K, const bf16 *V, int B, int L, int H, int D, int L_cap, bf16 *kc, bf16 *vt,
                           cudaStream_t st) {
  if (L <= 0) return cudaSuccess;
  dim3 grid(static_cast<unsigned>((static_cast<long long>(L) * D + 255) / 256), H, B);
  return launch_pdl(load_kv_kernel, dim3(grid), dim3(256), 0, st, K, V, L, H, D, L_cap, kc, vt);
}

}  // namespace fvar
