// Epilogues of the GEMM forms whose results arrive feature by feature: four features of a row a thread after a reduction
// through shared memory, or a warp's 32 features x 32 rows straight from TMEM (lane = feature).
#pragma once
#include "gemm_common.cuh"

namespace fvar {

__device__ __forceinline__ uint2 pack4_bf16(float a, float b, float c, float d) {
  return make_uint2(pack_bf16(a, b), pack_bf16(c, d));
}

// What the epilogue of (row, features n .. n + 3) reads besides the sums: fetched together with them, so that a row pays
// one memory latency and not two.
struct SkinnyFetch {
  float4 resid, gate;
  int jo;                  // output row within the element (after the scatter)
};
template <int EPI>
__device__ __forceinline__ SkinnyFetch skinny_fetch(const GemmArgs &p, int row, int n) {
  SkinnyFetch f;
  f.resid = f.gate = make_float4(0.f, 0.f, 0.f, 0.f);
  f.jo = 0;
  if constexpr (EPI == EPI_RESID) {
    const int e = row / p.rows_per_batch, j = row - e * p.rows_per_batch;
    f.resid = *reinterpret_cast<const float4 *>(p.resid + (static_cast<long long>(e * p.rmap.bmul + p.rmap.boff) * p.rmap.rpb + j) * p.ld_out + n);
    f.gate = resid_gate(p, e * p.bmul + p.boff, n);
    f.jo = p.scatter ? __ldg(p.scatter + static_cast<long long>(e) * p.rows_per_batch + j) : j;
  }
  return f;
}

// Epilogue of one thread for output row `row` (row of the flattened [R] rows), features n .. n + 3 (n % 4 == 0,
// n + 3 < N): the four sums arrive in `acc`.
template <int EPI>
__device__ __forceinline__ void skinny_store(const GemmArgs &p, float4 acc, const SkinnyFetch &f, int row, int n) {
  float v[4] = {acc.x, acc.y, acc.z, acc.w};
  if (p.bias != nullptr) {
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p.bias + n));
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
    const float2 f0 = __bfloat1622float2(h[0]), f1 = __bfloat1622float2(h[1]);
    v[0] += f0.x; v[1] += f0.y; v[2] += f1.x; v[3] += f1.y;
  }
  if constexpr (EPI == EPI_F32) {
    *reinterpret_cast<float4 *>(p.out_f32 + static_cast<long long>(row) * p.ld_out + n) = make_float4(v[0], v[1], v[2], v[3]);
  } else if constexpr (EPI == EPI_BF16 || EPI == EPI_GELU_BF16) {
    if constexpr (EPI == EPI_GELU_BF16) {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = gelu_tanh_f(v[i]);
    }
    *reinterpret_cast<uint2 *>(p.out_bf16 + static_cast<long long>(row) * p.ld_out + n) = pack4_bf16(v[0], v[1], v[2], v[3]);
  } else if constexpr (EPI == EPI_QKV) {
    const int e = row / p.rows_per_batch, j = row - e * p.rows_per_batch;
    const int b = e * p.bmul + p.boff;
    const int vc = n + p.col_base;
    if (vc < p.C) {
      *reinterpret_cast<uint2 *>(p.out_bf16 + static_cast<long long>(row) * p.ld_out + vc) = pack4_bf16(v[0], v[1], v[2], v[3]);
    } else if (vc < 2 * p.C) {
      const int c = vc - p.C, h = c / p.D, d0 = c - h * p.D;
      bf16 *dst = p.kc + ((static_cast<long long>(b) * p.H + h) * p.L_cap + p.L_prev + j) * p.D + d0;
      *reinterpret_cast<uint2 *>(dst) = pack4_bf16(v[0], v[1], v[2], v[3]);
    } else {
      const int c = vc - 2 * p.C, h = c / p.D, d0 = c - h * p.D;
      bf16 *dst = p.vt + ((static_cast<long long>(b) * p.H + h) * p.D + d0) * p.L_cap + p.L_prev + j;
#pragma unroll
      for (int i = 0; i < 4; ++i) dst[static_cast<long long>(i) * p.L_cap] = __float2bfloat16_rn(v[i]);
    }
  } else if constexpr (EPI == EPI_RESID) {
    const int e = row / p.rows_per_batch, jo = f.jo;
    const float4 r4 = f.resid, g4 = f.gate;
    v[0] = fmaf(g4.x, v[0], r4.x);
    v[1] = fmaf(g4.y, v[1], r4.y);
    v[2] = fmaf(g4.z, v[2], r4.z);
    v[3] = fmaf(g4.w, v[3], r4.w);
    *reinterpret_cast<float4 *>(p.out_f32 + (static_cast<long long>(e * p.omap.bmul + p.omap.boff) * p.omap.rpb + jo) * p.ld_out + n) =
        make_float4(v[0], v[1], v[2], v[3]);
    if (p.xsplit != nullptr) {
      bf16 *hi = p.xsplit + (static_cast<long long>(e) * 2 * p.xsplit_mk + jo) * p.ld_out + n;
      float lo[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) lo[i] = v[i] - __bfloat162float(__float2bfloat16_rn(v[i]));
      *reinterpret_cast<uint2 *>(hi) = pack4_bf16(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<uint2 *>(hi + static_cast<long long>(p.xsplit_mk) * p.ld_out) = pack4_bf16(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}

// Arg-max epilogue of one warp for output row `row`: lane l holds the sums of features n .. n + 3 of the 128-feature
// tile.  One packed word per row and tile leaves the warp (see GemmArgs::best).
__device__ __forceinline__ void skinny_argmax(const GemmArgs &p, float4 acc, int row, int n, int lane) {
  unsigned long long word = 0ull;                            // nothing: every real score packs to more
  if (n < p.N) {                                             // n % 4 == 0 and N % 8 == 0: all four or none
    const float4 h4 = __ldg(reinterpret_cast<const float4 *>(p.col_sub + n));
    word = argmax_word(acc.x - h4.x, n);
    word = max(word, argmax_word(acc.y - h4.y, n + 1));
    word = max(word, argmax_word(acc.z - h4.z, n + 2));
    word = max(word, argmax_word(acc.w - h4.w, n + 3));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) word = max(word, __shfl_xor_sync(0xffffffffu, word, o));
  if (lane == 0) atomicMax(p.best + row, word);
}

// Epilogue of one warp for the 32 features n0 .. n0 + 31 (N % 32 == 0), 32 rows at a time: lane l brings feature n0 + l of
// every row.  The values cross a staging tile so that they leave in row order, eight lanes a 128- or 64-byte segment;
// the transposed V cache takes them as they came, 32 consecutive rows a feature.
template <int EPI>
struct RowsEpilogue {
  const GemmArgs &p;
  const int n0, lane;
  const uint32_t stage;                // 32 x 132 bytes of shared memory of this warp
  const int range;                     // EPI_PARTIAL: K range
  const int row_end;                   // first row that is not this tile's
  float bias;                          // of this lane's feature
  __device__ __forceinline__ RowsEpilogue(const GemmArgs &args, int first_feature, uint32_t stage_addr, int l, int k_range, int end_row)
      : p(args), n0(first_feature), lane(l), stage(stage_addr), range(k_range), row_end(end_row) {
    bias = (p.bias != nullptr && n0 < p.N) ? __bfloat162float(p.bias[n0 + lane]) : 0.f;
  }
  // What the chunk of rows `row0` .. row0 + 31 reads besides its sums (EPI_RESID).
  struct Fetch {
    ResidRow rr;
    ResidPre pre;
  };
  __device__ __forceinline__ void prefetch(int row0, Fetch &f) const {
    if constexpr (EPI == EPI_RESID) {
      f.rr = resid_row(p, row0 + lane, row_end);
      resid_fetch(p, f.rr, n0, lane, f.pre);
    }
  }
  // acc[i] = sum of row row0 + i.
  __device__ __forceinline__ void chunk(const uint32_t (&acc)[32], int row0, const Fetch &f) const {
    const int vc0 = n0 + p.col_base;
    if (EPI == EPI_QKV && vc0 >= 2 * p.C) {              // uniform across the warp: C % 64 == 0
#pragma unroll
      for (int i = 0; i < 32; ++i)
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(stage + i * 132 + lane * 4), "f"(__uint_as_float(acc[i]) + bias) : "memory");
      __syncwarp();
      const int row = row0 + lane;
      if (row < row_end) {
        const int e = row / p.rows_per_batch, j = row - e * p.rows_per_batch, b = e * p.bmul + p.boff;
        const int c = vc0 - 2 * p.C, h = c / p.D, d0 = c - h * p.D;
        bf16 *dst = p.vt + ((static_cast<long long>(b) * p.H + h) * p.D + d0) * p.L_cap + p.L_prev + j;
#pragma unroll 8
        for (int f = 0; f < 32; ++f) {
          float v;
          asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(stage + lane * 132 + f * 4));
          dst[static_cast<long long>(f) * p.L_cap] = __float2bfloat16_rn(v);
        }
      }
      __syncwarp();
      return;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      float v = __uint_as_float(acc[i]) + bias;
      if constexpr (EPI == EPI_GELU_BF16) v = gelu_tanh_f(v);
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(stage + i * 128 + lane * 4), "f"(v) : "memory");
    }
    // where this lane's row of the chunk goes, for the lanes that will store it (EPI_QKV: element offset / D of K head 0)
    int k_off = 0;
    if constexpr (EPI == EPI_QKV) {
      const int row = row0 + lane, e = row / p.rows_per_batch, j = row - e * p.rows_per_batch;
      k_off = (e * p.bmul + p.boff) * p.H * p.L_cap + p.L_prev + j;
    }
    __syncwarp();
    const int c4 = lane & 7, n = n0 + c4 * 4, vc = vc0 + c4 * 4;
    const int ck = vc - p.C, hk = (EPI == EPI_QKV) ? ck / p.D : 0, dk = ck - hk * p.D;
    float4 v[8];                         // all of them, then the stores: neither waits for the other row by row
#pragma unroll
    for (int it = 0; it < 8; ++it) v[it] = ld_shared_f4(stage + (it * 4 + (lane >> 3)) * 128 + c4 * 16);
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      const int r = it * 4 + (lane >> 3), row = row0 + r;
      const float4 o = v[it];
      if constexpr (EPI == EPI_RESID) {
        resid_store(p, f.rr, o, f.pre, it, r, n);
      } else if constexpr (EPI == EPI_F32 || EPI == EPI_PARTIAL) {
        const int at = EPI == EPI_PARTIAL ? range * p.R + row : row;
        if (row < row_end) *reinterpret_cast<float4 *>(p.out_f32 + static_cast<long long>(at) * p.ld_out + n) = o;
      } else if constexpr (EPI == EPI_QKV) {
        const int ko = __shfl_sync(0xffffffffu, k_off, r);
        if (row < row_end) {
          bf16 *dst = vc0 < p.C ? p.out_bf16 + static_cast<long long>(row) * p.ld_out + vc
                                : p.kc + (static_cast<long long>(ko) + static_cast<long long>(hk) * p.L_cap) * p.D + dk;
          *reinterpret_cast<uint2 *>(dst) = pack4_bf16(o.x, o.y, o.z, o.w);
        }
      } else {
        if (row < row_end) *reinterpret_cast<uint2 *>(p.out_bf16 + static_cast<long long>(row) * p.ld_out + n) = pack4_bf16(o.x, o.y, o.z, o.w);
      }
    }
    __syncwarp();
  }
};

}  // namespace fvar
