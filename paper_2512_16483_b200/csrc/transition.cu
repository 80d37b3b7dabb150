// Kernels of the transition between two scale steps (the paper's Algorithm 1, "Vanilla VAR" lines;
// Eq. "var_upf", Eq. "var_downf"): R_k = Q(F_k^o), F_k = F_{k-1} + Up(R_k, (h_K, w_K)), next input =
// Down(F_k, (h_{k+1}, w_{k+1})).  Q is the nearest codeword: its scores F_k^o Z^T - |Z_v|^2 / 2 come from the
// tensor-core GEMM with the arg-max epilogue; the kernels here supply the half-norms, decode the winning
// columns, gather + upsample + accumulate the codewords (HBM-bound, 16-byte accesses) and average the
// accumulated map down to the next scale.
#include "internal.h"
#include "ptx.cuh"

namespace fvar {

// hn[v] = |Z_v|^2 / 2 in fp32: one warp per codeword.
__global__ void __launch_bounds__(256) half_norms_kernel(const bf16 *__restrict__ Z, int V, int C, float *__restrict__ hn) {
  const int v = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (v >= V) return;
  const uint4 *row = reinterpret_cast<const uint4 *>(Z + static_cast<long long>(v) * C);
  float acc = 0.f;
  for (int g = lane; g < C / 8; g += 32) {
    const uint4 u = __ldg(row + g);
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float2 f = __bfloat1622float2(h[t]);
      acc = fmaf(f.x, f.x, acc);
      acc = fmaf(f.y, f.y, acc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) hn[v] = 0.5f * acc;
}

cudaError_t launch_half_norms(const bf16 *Z, int V, int C, float *hn, cudaStream_t st) {
  if (V <= 0) return cudaSuccess;
  half_norms_kernel<<<(V + 7) / 8, 256, 0, st>>>(Z, V, C, hn);
  return cudaGetLastError();
}

// The winning column of a row out of its packed word (low half = ~column).  A row no tile wrote (word still zero)
// or a column out of range yields code 0.
__device__ __forceinline__ int code_of(unsigned long long word, int V, bool *bad) {
  const unsigned c = 0xFFFFFFFFu - static_cast<unsigned>(word & 0xFFFFFFFFull);
  *bad = (word == 0ull) || c >= static_cast<unsigned>(V);
  return *bad ? 0 : static_cast<int>(c);
}

// F[b][p][:] (+)= sum over the four bilinear neighbours of pixel p on the (h0, w0) grid of weight x
// Z[code of neighbour][:] (half-pixel centres, source coordinate clamped at 0, neighbours clamped at the
// edge: the library's Up).  One warp per target pixel; fp32 accumulator map.  C % 8 == 0.
// The codes are decoded from the arg-max words where they are used; the grid's threads also write them out for the
// caller, flag the status word for a bad one, and zero the words the next codeword search will use (`clear`: a second
// buffer, nobody's by now) -- in a chain of 3 us launches the memset, the unpacking kernel and the copy were half of
// the transition's launches.  Bound by the map (8 C bytes a pixel, from L2 while it fits) and the gathered
// codewords (as much again).  The map moves 32 bytes a lane: as two accesses of 16 each of them touched half of every sector
// it named, and the stores went to L2 as twice the masked halves (eleven transitions of one 64 x 64 map, C = 2048, 8192
// codewords 522 -> 478 us, 1024 codewords 406 -> 354; thirteen of four maps 2470 -> 2395; one round of loads in flight
// instead of four 517 and 380).  C % 8 == 0 and a map on a 32-byte grid (it is the workspace's).
__global__ void __launch_bounds__(256) up_accumulate_kernel(const bf16 *__restrict__ Z, const unsigned long long *__restrict__ best,
                                                            int V, int B, int h0, int w0, int h1, int w1, int C, int overwrite,
                                                            float *__restrict__ F, int *__restrict__ codes,
                                                            unsigned long long *__restrict__ clear, long long n_clear, unsigned *status) {
  pdl_wait();
  pdl_launch_dependents();
  const int M1 = h1 * w1;
  const long long n_codes = static_cast<long long>(B) * h0 * w0, nthreads = static_cast<long long>(gridDim.x) * blockDim.x;
  const long long tid = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  bool bad;
  for (long long i = tid; i < n_codes; i += nthreads) {
    const int c = code_of(best[i], V, &bad);
    if (bad) atomicOr(status, kStatusBadIndex);
    if (codes != nullptr) codes[i] = c;
  }
  for (long long i = tid; i < n_clear; i += nthreads) clear[i] = 0ull;
  const long long gw = tid >> 5;
  if (gw >= static_cast<long long>(B) * M1) return;
  const int b = static_cast<int>(gw / M1), i = static_cast<int>(gw - static_cast<long long>(b) * M1);
  const int y = i / w1, xq = i - y * w1;
  const BilinearTap tap = bilinear_tap(y, xq, h0, w0, h1, w1);
  const int y0 = tap.y0, y1 = tap.y1, x0 = tap.x0, x1 = tap.x1;
  const unsigned long long *wb = best + static_cast<long long>(b) * h0 * w0;
  auto row = [&](int yy, int xx) { return reinterpret_cast<const uint4 *>(Z + static_cast<long long>(code_of(__ldg(wb + yy * w0 + xx), V, &bad)) * C); };
  const uint4 *p00 = row(y0, x0), *p01 = row(y0, x1), *p10 = row(y1, x0), *p11 = row(y1, x1);
  const float w00 = tap.w00, w01 = tap.w01, w10 = tap.w10, w11 = tap.w11;
  float *dst = F + (static_cast<long long>(b) * M1 + i) * C;
#pragma unroll 4
  for (int g = threadIdx.x & 31; g < C / 8; g += 32) {
    const uint4 a = __ldg(p00 + g), bq = __ldg(p01 + g), cq = __ldg(p10 + g), d = __ldg(p11 + g);
    float prev[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (!overwrite) ld_global_32(dst + 8 * g, prev);
    const __nv_bfloat162 *ha = reinterpret_cast<const __nv_bfloat162 *>(&a), *hb = reinterpret_cast<const __nv_bfloat162 *>(&bq);
    const __nv_bfloat162 *hc = reinterpret_cast<const __nv_bfloat162 *>(&cq), *hd = reinterpret_cast<const __nv_bfloat162 *>(&d);
    uint32_t o[8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const float2 fa = __bfloat1622float2(ha[t]), fb = __bfloat1622float2(hb[t]);
      const float2 fc = __bfloat1622float2(hc[t]), fd = __bfloat1622float2(hd[t]);
      o[2 * t] = __float_as_uint(w00 * fa.x + w01 * fb.x + w10 * fc.x + w11 * fd.x + prev[2 * t]);
      o[2 * t + 1] = __float_as_uint(w00 * fa.y + w01 * fb.y + w10 * fc.y + w11 * fd.y + prev[2 * t + 1]);
    }
    st_global_32(dst + 8 * g, o);
  }
}

cudaError_t launch_up_accumulate(const bf16 *Z, const unsigned long long *best, int V, int B, int h0, int w0, int h1, int w1, int C,
                                 bool overwrite, float *F, int *codes, unsigned long long *clear, long long n_clear, unsigned *status,
                                 cudaStream_t st) {
  const long long warps = static_cast<long long>(B) * h1 * w1;
  if (warps <= 0) return cudaSuccess;
  if (C % 8 != 0) return cudaErrorInvalidValue;
  return launch_pdl(up_accumulate_kernel, dim3(static_cast<unsigned>((warps + 7) / 8)), dim3(256), 0, st, Z, best, V, B, h0, w0,
                    h1, w1, C, overwrite ? 1 : 0, F, codes, clear, n_clear, status);
}

// tokens[b][q][:] = mean of F over the source cells target cell q = (y, x) of the (h1, w1) grid covers:
// rows [floor(y h0 / h1), ceil((y + 1) h0 / h1)), columns likewise ("area" resampling); bf16 out.  C % 4 == 0.
// Two forms, chosen in launch_down_area.
//
// Few target cells, long windows: a thread owns four channels of one target cell; G groups of threads share the window's
// cells (group g takes cells g, g + G, ...) and their partial sums are added in group order through shared memory.  Bound
// by latency -- the map is in L2 then -- so G grows until about two thousand threads an SM are at work.
template <int G>
__global__ void __launch_bounds__(256) down_area_kernel(const float *__restrict__ F, int h0, int w0, int h1, int w1, int C, int slabs,
                                                        bf16 *__restrict__ tokens, int dup) {
  constexpr int kLanes = 256 / G;
  __shared__ float4 part[G > 1 ? 256 : 1];
  pdl_wait();
  pdl_launch_dependents();
  const int M1 = h1 * w1, b = blockIdx.y, q = blockIdx.x / slabs, slab = blockIdx.x - q * slabs;
  const int y = q / w1, x = q - y * w1;
  const int ya = (y * h0) / h1, yb = ((y + 1) * h0 + h1 - 1) / h1;
  const int xa = (x * w0) / w1, xb = ((x + 1) * w0 + w1 - 1) / w1;
  const int nx = xb - xa, cells = (yb - ya) * nx;
  const int grp = threadIdx.x / kLanes, c4 = slab * kLanes + threadIdx.x % kLanes;      // this thread's four channels
  const bool in = c4 < C / 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (in) {
    const float4 *src = reinterpret_cast<const float4 *>(F + static_cast<long long>(b) * h0 * w0 * C) + c4;
#pragma unroll 4
    for (int i = grp; i < cells; i += G) {
      const int yy = ya + i / nx, xx = xa + i % nx;
      const float4 v = __ldg(src + (static_cast<long long>(yy) * w0 + xx) * (C / 4));
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
  }
  if constexpr (G > 1) {
    part[threadIdx.x] = acc;
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int t = 1; t < G; ++t) {
      const float4 v = part[t * kLanes + threadIdx.x];
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
  }
  if (in) {
    const float inv = 1.0f / static_cast<float>(cells);
    const __nv_bfloat162 o0 = __floats2bfloat162_rn(acc.x * inv, acc.y * inv), o1 = __floats2bfloat162_rn(acc.z * inv, acc.w * inv);
    const uint2 pk = make_uint2(*reinterpret_cast<const uint32_t *>(&o0), *reinterpret_cast<const uint32_t *>(&o1));
    // dup: element b is written twice, as elements 2b and 2b + 1 (both branches of a CFG pair read the same tokens)
    uint2 *dst = reinterpret_cast<uint2 *>(tokens + (static_cast<long long>(dup ? 2 * b : b) * M1 + q) * C) + c4;
    dst[0] = pk;
    if (dup) dst[static_cast<long long>(M1) * C / 4] = pk;
  }
}

// Many target cells, short windows: a warp a cell with all channels, four groups of four channels a lane at a time, so
// that a block is eight whole cells and not a slice of one, whose start and end then cost more than its reads of 4 KB:
// eight elements of a 64 x 64 map to 64 x 64 tokens for both branches, 537 MB, 161 us in the other form, 88 in this one.
__global__ void __launch_bounds__(256) down_area_cells_kernel(const float *__restrict__ F, int B, int h0, int w0, int h1, int w1, int C,
                                                              bf16 *__restrict__ tokens, int dup) {
  pdl_wait();
  pdl_launch_dependents();
  const int M1 = h1 * w1, lane = threadIdx.x & 31;
  const long long cell = static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (cell >= static_cast<long long>(B) * M1) return;
  const int b = static_cast<int>(cell / M1), q = static_cast<int>(cell - static_cast<long long>(b) * M1);
  const int y = q / w1, x = q - y * w1;
  const int ya = (y * h0) / h1, yb = ((y + 1) * h0 + h1 - 1) / h1;
  const int xa = (x * w0) / w1, xb = ((x + 1) * w0 + w1 - 1) / w1;
  const float inv = 1.0f / static_cast<float>((yb - ya) * (xb - xa));
  const int n4 = C / 4;
  const float4 *src = reinterpret_cast<const float4 *>(F + static_cast<long long>(b) * h0 * w0 * C);
  uint2 *dst = reinterpret_cast<uint2 *>(tokens + (static_cast<long long>(dup ? 2 * b : b) * M1 + q) * C);
  for (int g0 = lane; g0 < n4; g0 += 128) {
    float4 acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int yy = ya; yy < yb; ++yy)
      for (int xx = xa; xx < xb; ++xx) {
        const float4 *cellp = src + (static_cast<long long>(yy) * w0 + xx) * n4;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (g0 + 32 * u < n4) {
            const float4 v = __ldg(cellp + g0 + 32 * u);
            acc[u].x += v.x; acc[u].y += v.y; acc[u].z += v.z; acc[u].w += v.w;
          }
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (g0 + 32 * u < n4) {
        const __nv_bfloat162 o0 = __floats2bfloat162_rn(acc[u].x * inv, acc[u].y * inv), o1 = __floats2bfloat162_rn(acc[u].z * inv, acc[u].w * inv);
        const uint2 pk = make_uint2(*reinterpret_cast<const uint32_t *>(&o0), *reinterpret_cast<const uint32_t *>(&o1));
        dst[g0 + 32 * u] = pk;
        if (dup) dst[static_cast<long long>(M1) * n4 + g0 + 32 * u] = pk;
      }
  }
}

template <int G>
static cudaError_t launch_down(const float *F, int B, int h0, int w0, int h1, int w1, int C, bf16 *tokens, bool dup, cudaStream_t st) {
  const int slabs = (C / 4 + 256 / G - 1) / (256 / G);
  return launch_pdl(down_area_kernel<G>, dim3(static_cast<unsigned>(h1 * w1 * slabs), B), dim3(256), 0, st, F, h0, w0, h1, w1, C, slabs, tokens, dup ? 1 : 0);
}

cudaError_t launch_down_area(const float *F, int B, int h0, int w0, int h1, int w1, int C, bf16 *tokens, bool dup, cudaStream_t st) {
  if (C % 4 != 0) return cudaErrorInvalidValue;
  if (B <= 0 || h1 <= 0 || w1 <= 0) return cudaSuccess;
  // A warp a cell walks a chain of (cells of a window) x (C / 512) rounds of loads, which it hides behind the other warps
  // only if there are many: it is taken from 160 warps a round on.  Whole chains of transitions (guidance, search, Up,
  // Down; 64 x 64 map, C = 2048, us), the line at 160 against the shared form alone: up to 40 x 40 cells, which that line
  // leaves to the shared form for one element, level (one 523 and 522, two 826 and 829, four 1513 and 1518, eight 2900 and
  // 2894); up to 64 x 64 one 734 and 748, two 1247 and 1275, four 2424 and 2523, eight 4902 and 5039.  Timed launch by
  // launch a warp a cell wins from 40 warps a round on (64 x 64 cells of one element 12 against 25 us, of eight 88 against
  // 161), but a line there costs in the chain: one element 536 and 747, two 843 and 1264.  For 2 x 2 cells it takes 1047 -
  // 1972 us, the other form 21 - 69.
  const double warps = static_cast<double>(B) * h1 * w1, rounds = static_cast<double>(h0) * w0 / (static_cast<double>(h1) * w1) * C / 512.0;
  if (warps >= 160.0 * rounds || B > 65535)        // 65535: rows of the other form's grid
    return launch_pdl(down_area_cells_kernel, dim3(static_cast<unsigned>((static_cast<long long>(B) * h1 * w1 + 7) / 8)), dim3(256), 0, st, F, B, h0, w0, h1, w1, C,
                      tokens, dup ? 1 : 0);
  const double threads = static_cast<double>(B) * h1 * w1 * (C / 4), cells = static_cast<double>(h0) * w0 / (static_cast<double>(h1) * w1);
  const double want = 300000.0 / threads < cells ? 300000.0 / threads : cells;      // groups for 148 x 2048 threads, at most one a cell
  if (want > 8.0) return launch_down<16>(F, B, h0, w0, h1, w1, C, tokens, dup, st);
  if (want > 2.0) return launch_down<4>(F, B, h0, w0, h1, w1, C, tokens, dup, st);
  return launch_down<1>(F, B, h0, w0, h1, w1, C, tokens, dup, st);
}

// Classifier-free guidance on CFG pairs: out[p] = null + s (prompt - null) with (prompt, null) = elements
// (2p, 2p + 1); fp32 arithmetic on bf16 inputs, one rounding.  Eight elements per thread.
__global__ void __launch_bounds__(256) cfg_combine_kernel(const bf16 *__restrict__ pair, long long n8_per_elem, long long total8,
                                                          float s, bf16 *__restrict__ out) {
  pdl_wait();
  pdl_launch_dependents();
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= total8) return;
  const long long pidx = i / n8_per_elem, off = i - pidx * n8_per_elem;
  const uint4 ua = __ldg(reinterpret_cast<const uint4 *>(pair) + (2 * pidx) * n8_per_elem + off);
  const uint4 ub = __ldg(reinterpret_cast<const uint4 *>(pair) + (2 * pidx + 1) * n8_per_elem + off);
  const __nv_bfloat162 *ha = reinterpret_cast<const __nv_bfloat162 *>(&ua), *hb = reinterpret_cast<const __nv_bfloat162 *>(&ub);
  uint32_t w[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const float2 a = __bfloat1622float2(ha[t]), b = __bfloat1622float2(hb[t]);
    const __nv_bfloat162 o = __floats2bfloat162_rn(fmaf(s, a.x - b.x, b.x), fmaf(s, a.y - b.y, b.y));
    w[t] = *reinterpret_cast<const uint32_t *>(&o);
  }
  reinterpret_cast<uint4 *>(out)[i] = make_uint4(w[0], w[1], w[2], w[3]);
}

cudaError_t launch_cfg_combine(const bf16 *pair, int pairs, long long per_elem, float s, bf16 *out, cudaStream_t st) {
  if (per_elem % 8 != 0) return cudaErrorInvalidValue;
  const long long total8 = static_cast<long long>(pairs) * (per_elem / 8);
  if (total8 <= 0) return cudaSuccess;
  return launch_pdl(cfg_combine_kernel, dim3(static_cast<unsigned>((total8 + 255) / 256)), dim3(256), 0, st, pair, per_elem / 8,
                    total8, s, out);
}

}  // namespace fvar
