// Flash-style attention of one scale's query rows over the multi-scale KV cache, sm_100a.
//
// One CTA handles up to 256 query rows (two tiles of 128) of one (batch element, head).
//   warp 0      streams K and V^T tiles of 128 keys through a ring of shared-memory slots (TMA);
//   warp 1      issues S_t = Q_t K^T and O_t += P_t V on the tensor cores, accumulators in TMEM;
//   warps 4-7   softmax of tile 0, one query row per thread;   warps 8-11: softmax of tile 1.
// The two tiles run out of phase: while one warp-group turns S into P (row max, exp2, bf16 P
// written back into the TMEM columns S came from), the tensor core works for the other tile (P V of
// block j, with P read from TMEM as the A operand, then Q K^T of block j+1).  P is handed over in two halves, so that
// P V starts on the first 64 keys while the exponentials of the others are still being taken.  Keeping P out of shared
// memory matters: the operand reads of the MMAs alone nearly fill the 128 B/clk of shared-memory
// bandwidth, and a P tile costs one write and one read on top.  O stays in TMEM for the whole key loop; its rows are rescaled only when the
// running maximum has grown by more than 2^8 since the last rescale, so the common case costs no
// TMEM round trip.  Keys at or beyond L are masked.
//
// What bounds it (B = 2, H = 16, D = 128, r = 4096, L = 10521, per key block and tile pair; 2048 clocks of MMA): before,
// the issuing thread was busy 3100 of 3576 clocks moving operands for 32 MMAs, one lane of a branch at a time; with
// predicated issue by the whole warp the MMAs alone take 2345 and the period is 3100, which is one tile's chain softmax
// (1800, of it 1413 exponentials) -> P V -> Q K^T (1188).  691 -> 584 us (1018 -> 1208 TFLOP/s).
// Every wait is bounded (see ptx.cuh).
//
// Few queries over a long cache (few CTAs, many key blocks): the key range is split over a thread-block cluster of
// up to 6 CTAs.  Each pushes its unnormalised rows (O, m, l) into its peers' shared memory; after a cluster barrier every
// CTA merges a slice of the query rows over all ranges, in range order (the result does not depend on timing),
// normalises and stores.  Nothing goes through global scratch.
#include <limits.h>
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace fvar {

constexpr int kAttnThreads = 384;
constexpr int kSoftmaxWarp = 4;            // first softmax warp: warp-group 0 holds the producer and the MMA issuer
constexpr int kRegsIssue = 72, kRegsSoftmax = 208;   // registers a thread after the split (see attention_prepare)
constexpr int kQRows = 128;
constexpr int kKeys = 128;
constexpr int kAtomBytes = 128 * 128;   // [128 rows][64 bf16] swizzled tile
constexpr float kRescaleThreshold = 8.0f;   // log2 units

// Softmax arithmetic on pairs of neighbouring keys: packed fp32, one instruction slot for two keys, and three-input
// maxima (a block took 576 issue slots a row, now 390).  Moving part of the exponentials from the special-function unit
// to a polynomial on the FMA pipe (degree 5, 1/8 to 1/2 of the keys) was measured and left out: 1144 TFLOP/s without,
// 1121 / 1089 / 1036 with 1/8, 1/4, 3/8 of them -- the chain through a tile's softmax bounds the kernel, not the unit.
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void unpack_f2(uint64_t v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

template <int D>
struct AttnCfg {
  static constexpr int kTileBytes = 128 * D * 2;          // a Q tile, a K tile [128 keys][D] or a V^T tile [D][128 keys]
  static constexpr int kRing = (D == 64) ? 10 : 5;        // K_j, V_j, K_{j+1}, ...
  static constexpr int kQBytes = 2 * kTileBytes;
  static constexpr int kSmemBytes = kQBytes + kRing * kTileBytes + 1024 + 256;
  // TMEM: S0 [0,128), S1 [128,256), O0 [256,256+D), O1 [256+D,256+2D).  P (bf16, two keys per 32-bit
  // column) overwrites columns [0,64) of the S buffer it was computed from.
  static constexpr int kTmemCols = 512;
  static_assert(kSmemBytes > 116 * 1024, "one CTA per SM (the CTA allocates all of TMEM)");
  static_assert(kSmemBytes + 64 <= 227 * 1024, "shared memory");
  static_assert(256 + 2 * D <= 512, "TMEM columns");
};

// u / d by one multiplication where that is exact (see launch_d), else by a division (two in each role's way were 0.9 us
// of a 6 us launch).
__device__ __forceinline__ int fast_div(int u, const FastDiv &f) {
  return f.mul ? static_cast<int>(__umulhi(static_cast<unsigned>(u), f.mul)) : u / static_cast<int>(f.d);
}

// How the units of work are spread over the grid: each CTA walks several, has one, or shares one with its cluster.
enum { kWalk = 0, kOne = 1, kRanges = 2 };

template <int D, int MODE, bool DUAL>
__global__ void __launch_bounds__(kAttnThreads, 1)
attention_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ AttnArgs p) {
  using Cfg = AttnCfg<D>;
  constexpr int NR = Cfg::kRing;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t tmem_base_holder;
  __shared__ volatile int abort_flag;

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t q_smem = smem_base;
  const uint32_t ring_smem = q_smem + Cfg::kQBytes;
  const uint32_t bar_base = ring_smem + NR * Cfg::kTileBytes;
  const uint32_t q_full = bar_base;
  const uint32_t q_empty = bar_base + 8u * (11 + 2 * NR);                 // every Q K^T of the unit has read Q
  auto ring_full = [&](int s) { return bar_base + 8u * (1 + s); };
  auto ring_empty = [&](int s) { return bar_base + 8u * (1 + NR + s); };
  auto s_full = [&](int t) { return bar_base + 8u * (1 + 2 * NR + t); };
  auto p_full = [&](int t) { return bar_base + 8u * (3 + 2 * NR + t); };
  auto o_full = [&](int t) { return bar_base + 8u * (5 + 2 * NR + t); };
  auto o_last = [&](int t) { return bar_base + 8u * (9 + 2 * NR + t); };   // P V of the last block
  auto p_half = [&](int t) { return bar_base + 8u * (7 + 2 * NR + t); };   // the first 64 keys of P are in TMEM

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wb = wait_budget(p.wait_cycles);
  // A unit of work: one or two query tiles of one (element, head) over one range of key blocks.  kRanges: the kv_splits
  // CTAs of a cluster take the key ranges of one unit each, grid (query tiles x ranges, H, elements); kOne: the same grid
  // without ranges; kWalk: a CTA walks the units blockIdx.x, blockIdx.x + gridDim.x, ...
  const int splits = MODE == kRanges ? p.kv_splits : 1;
  const int sp = MODE == kRanges ? static_cast<int>(blockIdx.x) % splits : 0;   // rank in the cluster
  const int tpc = p.tiles_per_cta == 1 ? 1 : 2;                   // query tiles a CTA takes: two, or one when CTAs are scarce
  const int unit0 = MODE == kWalk ? static_cast<int>(blockIdx.x) : 0, nunits = MODE == kWalk ? p.units : 1;
  const int unit_step = MODE == kWalk ? static_cast<int>(gridDim.x) : 1;
  const int nkv_total = (p.L + kKeys - 1) / kKeys;
  const int kv_per = MODE == kRanges ? (nkv_total + splits - 1) / splits : nkv_total;
  const int jb0 = sp * kv_per;                                    // first key block of this CTA
  const int nkv = min(kv_per, nkv_total - jb0);                   // >= 1: the host sizes splits so
  struct Unit {
    int q0, h, e, ntiles;                                         // first query row within the element; query tiles there are
  };
  auto unit_at = [&](int u) {
    Unit x;
    int qt;
    if constexpr (MODE != kWalk) {
      qt = static_cast<int>(blockIdx.x) / splits;
      x.h = blockIdx.y;
      x.e = blockIdx.z;
    } else {
      const int g = fast_div(u, p.div_nqt);                       // neighbouring units share keys and values (L2)
      qt = u - g * static_cast<int>(p.div_nqt.d);
      x.e = fast_div(g, p.div_h);
      x.h = g - x.e * p.H;
    }
    x.q0 = qt * tpc * kQRows;
    x.ntiles = (tpc == 2 && p.r - x.q0 > kQRows) ? 2 : 1;
    return x;
  };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    for (int s = 0; s < NR; ++s) {
      mbar_init(ring_full(s), 1);
      mbar_init(ring_empty(s), 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(s_full(t), 1);
      mbar_init(p_full(t), 128);
      mbar_init(p_half(t), 128);
      mbar_init(o_last(t), 1);
      mbar_init(o_full(t), 1);
    }
    mbar_fence_init();
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_holder), Cfg::kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  pdl_launch_dependents();      // the successor (a GEMM) only requests weights before its own wait
  // Tile i of a unit's stream of keys and values: K (v = 0) or V^T of which key block, and its request.
  auto stream_item = [&](int i, int &j, int &v) {
    j = i >> 1, v = i & 1;                         // even i: K of block i/2, odd i: V^T of block i/2
    if (DUAL) {                                    // K 0, K 1, V 0, K 2, V 1, K 3, ... V nkv-2, V nkv-1
      const int k = i - 2, alt = 2 * (nkv - 2);
      v = k >= alt || (k >= 0 && (k & 1) == 0);
      j = k < 0 ? i : k < alt ? (k >> 1) + (v ? 0 : 2) : k - alt + nkv - 2;
    }
  };
  auto request = [&](int slot, int j, int v, int bh) {
    mbar_expect_tx(ring_full(slot), Cfg::kTileBytes);
    const uint32_t dst = ring_smem + slot * Cfg::kTileBytes;
    if (v == 0) {
#pragma unroll
      for (int a = 0; a < D / 64; ++a) tma_load_3d(dst + a * kAtomBytes, &tmK, ring_full(slot), a * 64, (jb0 + j) * kKeys, bh);
    } else {
#pragma unroll
      for (int a = 0; a < 2; ++a) tma_load_3d(dst + a * (D * 128), &tmV, ring_full(slot), (jb0 + j) * kKeys + a * 64, 0, bh);
    }
  };
  // Tiles of the first unit that no kernel in flight writes are requested while the predecessor drains (see AttnArgs); as for the
  // weights of the GEMMs in a loop of their own, ahead of the producer's.
  int pre = 0;
  if (threadIdx.x == 0 && p.early_rows > 0) {
    const Unit x = unit_at(unit0);
    for (; pre < min(p.early_tiles, min(NR, 2 * nkv)); ++pre) {
      int j, v;
      stream_item(pre, j, v);
      if ((jb0 + j + 1) * kKeys > p.early_rows) break;
      request(pre, j, v, (x.e * p.bmul + p.boff) * p.H + x.h);
    }
  }
  pdl_wait();
  float m_ref = -INFINITY, l_run = 0.f;      // softmax threads: running maximum and sum of this thread's query row
  bool final_ok = false;                      // softmax threads: the last P V of the row's tile has completed

  if (warp < kSoftmaxWarp) {
  setmaxnreg_dec<kRegsIssue>();
  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------------- TMA producer
      uint32_t armed = (1u << pre) - 1u, last_parity = 0, q_units = 0;
      bool ok = true;
      int slot = pre == NR ? 0 : pre, first = pre;
      uint32_t phase = pre == NR ? 1u : 0u;
      for (int u = unit0; ok && u < nunits; u += unit_step) {
        const Unit x = unit_at(u);
        const int bh = (x.e * p.bmul + p.boff) * p.H + x.h;
        if (q_units > 0 && !mbar_wait(q_empty, (q_units - 1) & 1u, p.status, &abort_flag, wb)) { ok = false; break; }
        mbar_expect_tx(q_full, x.ntiles * Cfg::kTileBytes);
        for (int t = 0; t < x.ntiles; ++t)
#pragma unroll
          for (int a = 0; a < D / 64; ++a)
            tma_load_2d(q_smem + t * Cfg::kTileBytes + a * kAtomBytes, &tmQ, q_full, x.h * D + a * 64, x.e * p.r + x.q0 + t * kQRows);
        ++q_units;
        for (int i = first; i < 2 * nkv; ++i) {
          int j, v;
          stream_item(i, j, v);
          if (!mbar_wait(ring_empty(slot), phase ^ 1u, p.status, &abort_flag, wb)) { ok = false; break; }
          request(slot, j, v, bh);
          armed |= 1u << slot;
          last_parity = (last_parity & ~(1u << slot)) | (phase << slot);
          if (++slot == NR) { slot = 0; phase ^= 1u; }
        }
        first = 0;
      }
      if (!ok) {   // let every copy that was issued land before the shared memory is released
        const long long t0 = clock64();
        while (q_units > 0 && !mbar_try_wait(q_full, (q_units - 1) & 1u) && clock64() - t0 < kWaitCycles) {}
        for (int s = 0; s < NR; ++s)
          if (armed & (1u << s)) {
            const long long t1 = clock64();
            while (!mbar_try_wait(ring_full(s), (last_parity >> s) & 1u) && clock64() - t1 < kWaitCycles) {}
          }
      }
    }
  } else if (warp == 1) {
    {
      // ---------------------------------------------------------------- MMA issuer
      // The whole warp walks the loop; one elected lane issues (see umma_bf16_if).
      constexpr uint32_t idesc_s = umma_idesc_bf16(kQRows, kKeys);
      constexpr uint32_t idesc_o = umma_idesc_bf16(kQRows, D);
      const uint32_t leader = elect_one() ? 1u : 0u;
      auto wait = [&](uint32_t bar, uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, p.status, &abort_flag, wb)) != 0; };
      const uint64_t q_desc = smem_desc_sw128(q_smem), ring_desc = smem_desc_sw128(ring_smem);
      auto issue_s = [&](int t, int buf, int slot) {   // S buffer `buf` = Q_t K^T
        const uint64_t dq = q_desc + static_cast<uint32_t>(t * (Cfg::kTileBytes >> 4)), dk = ring_desc + static_cast<uint32_t>(slot * (Cfg::kTileBytes >> 4));
        const uint32_t ts = tmem_base + buf * kKeys;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) {
          constexpr uint32_t kAtom = kAtomBytes >> 4;
          umma_bf16_if(leader, ts, dq + ((k / 4) * kAtom + 2 * (k % 4)), dk + ((k / 4) * kAtom + 2 * (k % 4)), idesc_s, k != 0);
        }
        umma_commit_if(leader, s_full(buf));
      };
      // O_t (+)= P V over one half of the block's keys, P in S buffer `pbuf`
      auto issue_pv = [&](int t, int pbuf, int slot, int half, bool accumulate, bool last = false) {
        const uint64_t dv = ring_desc + static_cast<uint32_t>(slot * (Cfg::kTileBytes >> 4) + half * ((D * 128) >> 4));
        const uint32_t to = tmem_base + 256 + t * D, tp = tmem_base + pbuf * kKeys + 8 * half * (kKeys / 32);
#pragma unroll
        for (int k = 0; k < kKeys / 32; ++k)             // 16 keys of P = 8 columns of TMEM (two bf16 per column)
          umma_bf16_tmem_a_if(leader, to, tp + 8 * k, dv + 2 * k, idesc_o, (accumulate || k != 0) ? 1u : 0u);
        if (half == 1) umma_commit_if(leader, last ? o_last(t) : o_full(t));
      };
      // Phase parities: every barrier is waited for once per use, in order, so a bit per S / P buffer carries over from
      // unit to unit (pbits); within a unit the number of uses is known.
      bool ok = true;
      uint32_t pbits = 0, unit_parity = 0;
      unsigned base = 0;                                 // ring position of the unit's first K tile
      auto full = [&](unsigned idx) { return wait(ring_full(idx % NR), (idx / NR) & 1u); };
      for (int u = unit0; ok && u < nunits; u += unit_step, base += 2u * nkv) {
        const int ntiles = unit_at(u).ntiles;
        ok = wait(q_full, unit_parity) && full(base);
        unit_parity ^= 1u;
        if (!ok) break;
        tc_fence_after();
        for (int t = 0; t < ntiles; ++t) issue_s(t, t, base % NR);
        umma_commit_if(leader, ring_empty(base % NR));
        if (nkv == 1) umma_commit_if(leader, q_empty);
        if (DUAL) {
          // one tile, two streams of key blocks: stream t owns S buffer t, accumulator t and the blocks t, t + 2, ...
          unsigned pos = base + 1;
          if (!full(pos)) { ok = false; break; }
          tc_fence_after();
          issue_s(0, 1, pos % NR);
          umma_commit_if(leader, ring_empty(pos % NR));
          if (nkv == 2) umma_commit_if(leader, q_empty);
          ++pos;
          for (int j = 0; j < nkv; ++j) {
            const int t = j & 1;
            const uint32_t par = ((pbits >> t) ^ (j >> 1)) & 1u;
            if (!wait(p_half(t), par) || !full(pos)) { ok = false; break; }
            tc_fence_after();
            issue_pv(t, t, pos % NR, 0, j > 1);
            if (!wait(p_full(t), par)) { ok = false; break; }
            tc_fence_after();
            issue_pv(t, t, pos % NR, 1, true, j + 2 >= nkv);
            umma_commit_if(leader, ring_empty(pos % NR));
            ++pos;
            if (j + 2 < nkv) {
              if (!full(pos)) { ok = false; break; }
              tc_fence_after();
              issue_s(0, t, pos % NR);
              umma_commit_if(leader, ring_empty(pos % NR));
              if (j + 3 == nkv) umma_commit_if(leader, q_empty);
              ++pos;
            }
          }
          pbits ^= (((nkv + 1) >> 1) & 1u) | (((nkv >> 1) & 1u) << 1);
        } else if (ntiles == 1) {
          // A single query tile has no partner to alternate with: the idle tile's S columns serve as
          // a second S buffer, so that Q K^T of block j+1 runs while the softmax works on block j.  The idle tile's P
          // barriers alternate with its own too: the softmax may be done with block j+1 while this thread still waits
          // for the values of block j.
          for (int j = 0; j < nkv; ++j) {
            const unsigned vi = base + 2 * j + 1, ki = vi + 1;
            const int buf = j & 1;
            const uint32_t par = ((pbits >> buf) ^ (j >> 1)) & 1u;
            if (j + 1 < nkv) {
              if (!full(ki)) { ok = false; break; }
              tc_fence_after();
              issue_s(0, buf ^ 1, ki % NR);
              umma_commit_if(leader, ring_empty(ki % NR));
              if (j + 2 == nkv) umma_commit_if(leader, q_empty);
            }
            if (!wait(p_half(buf), par) || !full(vi)) { ok = false; break; }
            tc_fence_after();
            issue_pv(0, buf, vi % NR, 0, j > 0);
            if (!wait(p_full(buf), par)) { ok = false; break; }
            tc_fence_after();
            issue_pv(0, buf, vi % NR, 1, true, j + 1 == nkv);
            umma_commit_if(leader, ring_empty(vi % NR));
          }
          pbits ^= (((nkv + 1) >> 1) & 1u) | (((nkv >> 1) & 1u) << 1);
        } else {
          for (int j = 0; ok && j < nkv; ++j) {
            const unsigned vi = base + 2 * j + 1, ki = vi + 1;
            for (int t = 0; t < 2; ++t) {
              const uint32_t par = ((pbits >> t) ^ j) & 1u;
              if (!wait(p_half(t), par) || (t == 0 && !full(vi))) { ok = false; break; }
              tc_fence_after();
              issue_pv(t, t, vi % NR, 0, j > 0);
              if (!wait(p_full(t), par)) { ok = false; break; }
              tc_fence_after();
              issue_pv(t, t, vi % NR, 1, true, j + 1 == nkv);
              if (t == 1) umma_commit_if(leader, ring_empty(vi % NR));
              if (j + 1 < nkv) {
                if (t == 0 && !full(ki)) { ok = false; break; }
                tc_fence_after();
                issue_s(t, t, ki % NR);
                if (t == 1) {
                  umma_commit_if(leader, ring_empty(ki % NR));
                  if (j + 2 == nkv) umma_commit_if(leader, q_empty);
                }
              }
            }
          }
          pbits ^= (nkv & 1) ? 3u : 0u;
        }
      }
    }
  }
  } else {
    // ------------------------------------------------------------------ softmax warp-groups
    setmaxnreg_inc<kRegsSoftmax>();
    const int t = (warp - kSoftmaxWarp) >> 2;                       // query tile of this warp-group
    const int quad = warp & 3;                           // TMEM lanes [32 * quad, 32 * quad + 32)
    const int row_local = quad * 32 + lane;
    const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
    const uint32_t s_base = tmem_base + lane_addr;
    const uint32_t o_addr = tmem_base + 256 + t * D + lane_addr;
    const float c = p.scale_log2;
    uint32_t sbits = 0;                                  // parity of both S buffers at the start of the unit
    uint32_t o_bit = 0, last_bit = 0, unit_bit = 0;      // the same for this tile's o_full and o_last, and for o_last(0)
    bool ok = true;
    for (int u = unit0; ok && u < nunits; u += unit_step) {
      const int ntiles = unit_at(u).ntiles;
      const bool single = (ntiles == 1) && !DUAL;               // then S alternates between the two S buffers
      m_ref = -INFINITY;
      l_run = 0.f;
      const int nblk = DUAL ? (nkv + 1 - t) >> 1 : nkv;   // blocks of this warp-group: all, or those of its stream
      for (int j = 0; (DUAL || t < ntiles) && j < nblk; ++j) {
        const int sbuf = single ? (j & 1) : t;
        const uint32_t s_addr = s_base + sbuf * kKeys;
        ok = __all_sync(0xffffffffu, mbar_wait(s_full(sbuf), ((sbits >> sbuf) ^ (single ? (j >> 1) : j)) & 1u, p.status, &abort_flag, wb));
        if (!ok) break;
        tc_fence_after();
        const int valid = p.L - (jb0 + (DUAL ? 2 * j + t : j)) * kKeys;       // keys of this block below L (>= 128: all)
        // the whole S row (128 fp32) in registers: four TMEM loads in flight, one wait
        uint32_t v[4][32];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) tmem_ld32(s_addr + cc * 32, v[cc]);
        tmem_ld_wait();
        if (valid < kKeys) {                             // last block: mask keys at or beyond L
#pragma unroll
          for (int cc = 0; cc < 4; ++cc)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (cc * 32 + i >= valid) v[cc][i] = 0xff800000u;   // -inf
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int cc = 0; cc < 4; ++cc)
#pragma unroll
          for (int i = 0; i < 32; i += 2) mx[(i >> 1) & 3] = max3(mx[(i >> 1) & 3], __uint_as_float(v[cc][i]), __uint_as_float(v[cc][i + 1]));
        const float m_blk = fmaxf(max3(mx[0], mx[1], mx[2]), mx[3]);
        const float m_cand = fmaxf(m_ref, m_blk);
        const bool need = (m_cand - m_ref) * c > kRescaleThreshold;      // true on the first block (m_ref = -inf)
        if (__any_sync(0xffffffffu, need)) {
          if (j > 0) {
            // O is about to be touched: P V of block j-1 must be complete.  (P's own buffer is free in any case: the
            // S of this block was issued after the P V that last read it.  Waiting here on every block put the whole
            // P V of a lone tile into the chain softmax -> P V -> softmax.)
            ok = __all_sync(0xffffffffu, mbar_wait(o_full(t), (o_bit ^ (j - 1)) & 1u, p.status, &abort_flag, wb));
            if (!ok) break;
            tc_fence_after();
          }
          const float alpha = need ? exp2f((m_ref - m_cand) * c) : 1.0f;
          if (need) m_ref = m_cand;
          l_run *= alpha;
          if (j > 0) {
#pragma unroll 1
            for (int cc = 0; cc < D / 32; ++cc) {
              uint32_t o[32];
              tmem_ld32(o_addr + cc * 32, o);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
              tmem_st32(o_addr + cc * 32, o);
            }
            tmem_st_wait();
          }
        }
        const float neg_mc = -m_ref * c;
        const uint64_t c2 = pack_f2(c, c), neg_mc2 = pack_f2(neg_mc, neg_mc);
        uint64_t ls[2] = {0ull, 0ull};                   // packed zeros
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          // keys 32 * cc .. 32 * cc + 31 of this row, two per word: 16 TMEM columns.  The whole S row is in registers by
          // now, so overwriting its first columns loses nothing.
          uint32_t pk[16];
#pragma unroll
          for (int pr = 0; pr < 16; ++pr) {
            float p0, p1;
            unpack_f2(fma_f2(pack_f2(__uint_as_float(v[cc][2 * pr]), __uint_as_float(v[cc][2 * pr + 1])), c2, neg_mc2), p0, p1);
            p0 = exp2f(p0);                            // exp2(-inf) = 0 for masked keys
            p1 = exp2f(p1);
            ls[pr & 1] = add_f2(ls[pr & 1], pack_f2(p0, p1));
            __nv_bfloat162 v2 = __floats2bfloat162_rn(p0, p1);
            pk[pr] = *reinterpret_cast<uint32_t *>(&v2);
          }
          tmem_st16(s_addr + cc * 16, pk);
          if (cc & 1) {
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(cc == 1 ? p_half(sbuf) : p_full(sbuf));
          }
        }
        float l0, l1;
        unpack_f2(add_f2(ls[0], ls[1]), l0, l1);
        l_run += l0 + l1;
      }
      if (DUAL || t < ntiles) {
        // a barrier of its own: the blocks' o_full phases have not been waited for one by one, so their parity is no
        // safe guide here
        ok = ok && __all_sync(0xffffffffu, mbar_wait(o_last(t), last_bit, p.status, &abort_flag, wb));
        final_ok = ok;
        const uint32_t swap = q_smem + Cfg::kTileBytes + row_local * 8;
        if constexpr (DUAL) {
          // The two streams meet: a row's maximum and sum change sides through shared memory (the second query tile's room,
          // which no lone unit has), and each warp-group finishes half of the columns from both accumulators.  The barrier
          // carries the outcome of the waits: either all eight warps go on or none.
          asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(swap + t * (kQRows * 8)), "f"(m_ref), "f"(l_run) : "memory");
          ok = ok && __all_sync(0xffffffffu, mbar_wait(o_last(t ^ 1), last_bit, p.status, &abort_flag, wb));
          ok = bar_and(1, 256, ok);
        }
        if (MODE != kRanges && ok) {
          tc_fence_after();
          int u2 = u;                                    // decoded again: kept in registers through the loop, the unit spills
          asm volatile("" : "+r"(u2));
          const Unit x = unit_at(u2);
          const int rib = x.q0 + (DUAL ? 0 : t * kQRows) + row_local;
          bf16 *dst = p.out + (static_cast<long long>(x.e) * p.r + rib) * (p.H * D) + x.h * D;
          float inv_l, other = 0.f;
          if constexpr (DUAL) {
            const float2 ml = ld_shared_f2(swap + (t ^ 1) * (kQRows * 8));
            const float m_all = fmaxf(m_ref, ml.x), w0 = exp2f((m_ref - m_all) * c), w1 = exp2f((ml.x - m_all) * c);
            const float l_all = t == 0 ? fmaf(l_run, w0, ml.y * w1) : fmaf(ml.y, w1, l_run * w0);   // the same sum on both sides
            inv_l = w0 / l_all;
            other = w1 / l_all;
          } else {
            inv_l = 1.0f / l_run;
          }
          constexpr int kCols = DUAL ? D / 64 : D / 32;
          const int cc0 = DUAL ? t * kCols : 0;
          const bool wide = (reinterpret_cast<uintptr_t>(p.out) & 31) == 0;
#pragma unroll 1
          for (int cc = cc0; cc < cc0 + kCols; ++cc) {
            uint32_t v[32];
            tmem_ld32(o_addr + cc * 32, v);
            tmem_ld_wait();
            if constexpr (DUAL) {
              uint32_t v1[32];
              tmem_ld32(o_addr + (t == 0 ? D : -D) + cc * 32, v1);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(fmaf(__uint_as_float(v1[i]), other, __uint_as_float(v[i]) * inv_l));
            }
            if (rib < p.r) {
              const float norm = DUAL ? 1.f : inv_l;
              uint32_t w[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                __nv_bfloat162 v2 = __floats2bfloat162_rn(__uint_as_float(v[i * 2]) * norm, __uint_as_float(v[i * 2 + 1]) * norm);
                w[i] = *reinterpret_cast<uint32_t *>(&v2);
              }
              // every lane has a row of its own: the wider the store, the fewer passes over 32 lines each
              if (wide) {
                st_global_32(dst + cc * 32, w);
                st_global_32(dst + cc * 32 + 16, w + 8);
              } else {
#pragma unroll
                for (int q = 0; q < 4; ++q) reinterpret_cast<uint4 *>(dst + cc * 32)[q] = make_uint4(w[q * 4], w[q * 4 + 1], w[q * 4 + 2], w[q * 4 + 3]);
              }
            }
          }
        }
        // nobody hands over a P of the next unit, and so lets an accumulator be overwritten, before both halves are out
        if constexpr (MODE == kWalk && DUAL) {
          if (ok) asm volatile("bar.sync 1, 256;" ::: "memory");
        }
        o_bit ^= (nblk - 1) & 1u;
        last_bit ^= 1u;
      } else {
        // a unit with one tile uses both S buffers: its end is awaited, or the parity of the next wait would be ambiguous
        ok = __all_sync(0xffffffffu, mbar_wait(o_last(0), unit_bit, p.status, &abort_flag, wb));
        final_ok = ok;
      }
      unit_bit ^= 1u;
      sbits ^= single || DUAL ? ((((nkv + 1) >> 1) & 1u) | (((nkv >> 1) & 1u) << 1)) : ((nkv & 1) ? 3u : 0u);
    }
  }

  if constexpr (MODE == kRanges) {
    // ---------------------------------------------------------------- merge of the key ranges over the cluster
    // Row slice c of a tile is merged by CTA c.  Every CTA pushes its unnormalised rows (O, m, l) into the shared memory
    // of the slices' owners, where they are read locally: remote stores are not waited for one by one, as the remote
    // loads of the first form were (two dependent rounds of them a row: r = 400 over 2921 keys in two ranges 23.7 -> 20.9 us).  Every thread of every CTA of the
    // cluster passes the same barriers, whatever happened to its waits.
    const Unit x = unit_at(unit0);
    constexpr uint32_t kPitch = (D + 4) * 4;                       // bytes per row: conflict-free 16-byte accesses
    const int rpr0 = (min(kQRows, p.r - x.q0) + splits - 1) / splits;               // rows of a slice: tile 0 ...
    const int rpr1 = x.ntiles > 1 ? (min(kQRows, p.r - x.q0 - kQRows) + splits - 1) / splits : 0;   // ... and tile 1
    const int nrows = splits * (rpr0 + rpr1);                      // rows that arrive here, [tile][range][slice row]
    const uint32_t part_o = ring_smem, part_m = part_o + static_cast<uint32_t>(nrows) * kPitch;     // then maxima and sums
    tc_fence_before();
    cluster_sync_all();                                            // nobody's ring is in use any more
    if (warp >= kSoftmaxWarp && final_ok) {
      tc_fence_after();
      // A lone tile is shared by both warp-groups, half of the columns each.  Worth 0.4 % of a step of few rows with the merge below,
      // which is then not waited for (16 rows of 2048 columns 2538 -> 2526 us, 64 rows 2798 -> 2790), nothing without it.
      const int wg = (warp - kSoftmaxWarp) >> 2, t = x.ntiles > 1 ? wg : 0, row = (warp & 3) * 32 + lane, rpr = t == 0 ? rpr0 : rpr1;
      const int half = x.ntiles > 1 ? D / 32 : D / 64, cc0 = x.ntiles > 1 ? 0 : wg * half;
      const uint32_t o_addr = tmem_base + 256 + t * D + (static_cast<uint32_t>((warp & 3) * 32) << 16);
      const bool mine = x.q0 + t * kQRows + row < p.r;
      const int owner = mine ? row / rpr : 0, slot = (t == 0 ? 0 : splits * rpr0) + sp * rpr + row - owner * rpr;
      const uint32_t dst = mapa_shared(part_o + static_cast<uint32_t>(slot) * kPitch, static_cast<uint32_t>(owner));
      const uint32_t dst_m = mapa_shared(part_m + static_cast<uint32_t>(slot) * 8u, static_cast<uint32_t>(owner));
#pragma unroll 1
      for (int cc = cc0; cc < cc0 + half; ++cc) {
        uint32_t v[32];
        tmem_ld32(o_addr + cc * 32, v);
        tmem_ld_wait();
        if (mine) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (cc * 32 + q * 4) * 4), "r"(v[q * 4]), "r"(v[q * 4 + 1]),
                         "r"(v[q * 4 + 2]), "r"(v[q * 4 + 3]) : "memory");
        }
      }
      if (mine && t == wg) asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst_m), "f"(m_ref), "f"(l_run) : "memory");
    }
    tc_fence_before();
    cluster_sync_all();                                            // all rows have arrived; nobody touches a peer after this
    if (warp >= kSoftmaxWarp && abort_flag == 0) {
      constexpr int G = D / 4;                                     // threads per row, one float4 each
      const int st = static_cast<int>(threadIdx.x) - 32 * kSoftmaxWarp, d4 = (st % G) * 4;
      const float c = p.scale_log2;
#pragma unroll 1
      for (int k0 = 0; k0 < rpr0 + rpr1; k0 += 256 / G) {            // every lane of a warp goes round as often
        const bool there = k0 + st / G < rpr0 + rpr1;
        const int k = there ? k0 + st / G : 0;
        const int tt = k < rpr0 ? 0 : 1, lrow = tt == 0 ? k : k - rpr0, rpr = tt == 0 ? rpr0 : rpr1;
        const int rib = x.q0 + tt * kQRows + sp * rpr + lrow;
        const bool live = there && rib < p.r && sp * rpr + lrow < kQRows;
        const uint32_t slot0 = static_cast<uint32_t>((tt == 0 ? 0 : splits * rpr0) + lrow);
        // A lane of the row's threads takes one range's maximum and sum; the weights are formed side by side and handed round
        // (eight ranges at most), and the sum is the same whatever the timing.  One range after another in every thread, in two
        // passes, was a chain of 640 clocks a row (a step of 16 rows of 2048 columns 2544 -> 2538 us, of 64 rows 2818 -> 2798; 26 - 410
        // rows, in two ranges, level).  Code that runs once a launch has to be short: two rows a round cost 1.2 us of a
        // 21 us launch instead of gaining.
        const int l8 = st & 7;
        const float2 ml = l8 < splits ? ld_shared_f2(part_m + (slot0 + l8 * rpr) * 8u) : make_float2(-INFINITY, 0.f);
        float m_all = ml.x;
#pragma unroll
        for (int o2 = 4; o2 > 0; o2 >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(0xffffffffu, m_all, o2));
        float w8 = exp2f((ml.x - m_all) * c), l_all = ml.y * w8;
#pragma unroll
        for (int o2 = 4; o2 > 0; o2 >>= 1) l_all += __shfl_xor_sync(0xffffffffu, l_all, o2);
        w8 *= 1.0f / l_all;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t2 = 0; t2 < splits; ++t2) {
          const float w = __shfl_sync(0xffffffffu, w8, t2, 8);
          const float4 v = ld_shared_f4(part_o + (slot0 + t2 * rpr) * kPitch + d4 * 4);
          o.x = fmaf(w, v.x, o.x); o.y = fmaf(w, v.y, o.y); o.z = fmaf(w, v.z, o.z); o.w = fmaf(w, v.w, o.w);
        }
        if (!live) continue;
        __nv_bfloat162 h0 = __floats2bfloat162_rn(o.x, o.y), h1 = __floats2bfloat162_rn(o.z, o.w);
        *reinterpret_cast<uint2 *>(p.out + (static_cast<long long>(x.e) * p.r + rib) * (p.H * D) + x.h * D + d4) =
            make_uint2(*reinterpret_cast<uint32_t *>(&h0), *reinterpret_cast<uint32_t *>(&h1));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, Cfg::kTmemCols);
  }
}

template <int D, int MODE, bool DUAL>
static cudaError_t set_attr() {
  static bool attr_set = false;
  if (attr_set) return cudaSuccess;
  // The register split draws on what the block was launched with: refuse a build whose kernel got fewer.
  cudaFuncAttributes fa;
  cudaError_t err = cudaFuncGetAttributes(&fa, attention_kernel<D, MODE, DUAL>);
  if (err != cudaSuccess) return err;
  if (kAttnThreads * fa.numRegs < 32 * kSoftmaxWarp * kRegsIssue + (kAttnThreads - 32 * kSoftmaxWarp) * kRegsSoftmax) return cudaErrorInvalidConfiguration;
  err = cudaFuncSetAttribute(attention_kernel<D, MODE, DUAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnCfg<D>::kSmemBytes);
  if (err == cudaSuccess) attr_set = true;
  return err;
}

static int g_max_clusters[9];       // resident clusters of s CTAs (0: not asked or not launchable); the same for both widths: one CTA an SM

template <int D>
static cudaError_t set_attrs() {
  cudaError_t e = set_attr<D, kWalk, false>();
  if (e == cudaSuccess) e = set_attr<D, kWalk, true>();
  if (e == cudaSuccess) e = set_attr<D, kOne, false>();
  if (e == cudaSuccess) e = set_attr<D, kOne, true>();
  if (e == cudaSuccess) e = set_attr<D, kRanges, false>();
  return e;
}

cudaError_t attention_prepare() {
  cudaError_t e = set_attrs<64>();
  if (e == cudaSuccess) e = set_attrs<128>();
  if (e != cudaSuccess || g_max_clusters[1] > 0) return e;
  for (int s = 8; s >= 1; --s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(s * 64);
    cfg.blockDim = dim3(kAttnThreads);
    cfg.dynamicSmemBytes = AttnCfg<128>::kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = s;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attention_kernel<128, kRanges, false>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    g_max_clusters[s] = n;
  }
  return cudaSuccess;
}

static FastDiv make_fast_div(unsigned d, unsigned long long max_u) {
  // ceil(2^32 / d) is exact for u with u * d < 2^32; d == 1 does not fit 32 bits
  return FastDiv{d, (d > 1 && max_u * d < (1ull << 32)) ? static_cast<unsigned>(((1ull << 32) + d - 1) / d) : 0u};
}

template <int D, bool DUAL>
static cudaError_t launch_d(const CUtensorMap &tmQ, const CUtensorMap &tmK, const CUtensorMap &tmV, AttnArgs a, int num_sms,
                            cudaStream_t st) {
  using Cfg = AttnCfg<D>;
  const int nqt = (a.r + (a.tiles_per_cta == 1 ? 1 : 2) * kQRows - 1) / ((a.tiles_per_cta == 1 ? 1 : 2) * kQRows);
  const long long units = static_cast<long long>(nqt) * a.H * a.B_eff;
  if (units > INT_MAX) return cudaErrorInvalidValue;
  if (a.kv_splits <= 1 && units <= num_sms) {
    // the walk's bookkeeping is 0.5 us of a 4 us launch
    cudaError_t err = set_attr<D, kOne, DUAL>();
    if (err != cudaSuccess) return err;
    return launch_pdl(attention_kernel<D, kOne, DUAL>, dim3(nqt, a.H, a.B_eff), dim3(kAttnThreads), Cfg::kSmemBytes, st, tmQ, tmK, tmV, a);
  }
  if (a.kv_splits <= 1) {
    // one CTA an SM, each walking its share of the units: the set-up and first operands of a unit hide behind the last
    // blocks of the one before (D = 128: B = 2, r = 4096 over 256 context keys 42.3 -> 29.2 us; D = 64: B = 32, H = 30,
    // r = 128 over 552 keys 70.6 -> 48.7)
    cudaError_t err = set_attr<D, kWalk, DUAL>();
    if (err != cudaSuccess) return err;
    a.units = static_cast<int>(units);
    a.div_nqt = make_fast_div(nqt, units);
    a.div_h = make_fast_div(a.H, units);
    return launch_pdl(attention_kernel<D, kWalk, DUAL>, dim3(num_sms), dim3(kAttnThreads), Cfg::kSmemBytes, st, tmQ, tmK, tmV, a);
  }
  cudaError_t err = set_attr<D, kRanges, false>();
  if (err != cudaSuccess) return err;
  if (a.kv_splits > 8) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nqt * a.kv_splits, a.H, a.B_eff);
  cfg.blockDim = dim3(kAttnThreads);
  cfg.dynamicSmemBytes = Cfg::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;            // the key ranges of one query tile pair form a cluster
  attr[0].val.clusterDim.x = a.kv_splits;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = one_predecessor(st) ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, attention_kernel<D, kRanges, false>, tmQ, tmK, tmV, a);
}

// Launch shape of an attention call: query tiles per CTA (two: each K / V block feeds two tiles, the softmax of one
// overlapping the MMAs of the other; one: twice the units when there are few) and key ranges per unit (a cluster of up
// to 6 CTAs).  The pair with the least estimated time wins.  The estimate (microseconds) is fitted to forced launches of
// 21 shapes on B200, r = 16 .. 4096 over 55 .. 10521 keys, which it ranks as measured: a block of 128 keys takes a
// tile pair 1.6 and a lone tile 1.0 (0.85 as two streams); a unit 4 or 3 more for its own first operands and store; a launch 3.5; ranges pay
// for their set-up, the barriers and the rows that cross the cluster, and 4 more for each wave after the first (a new
// cluster starts only when all of its SMs are free).  Resident clusters come from the occupancy query, which a probe
// confirmed to the cluster (74 / 45 / 33 / 26 / 22 of 2 .. 6 CTAs, but 15 of 7 or 8, hence the limit).
constexpr int kMaxRanges = 6;

// A launch of lone query tiles without ranges has both warp-groups on each tile, one on every other key block: two streams
// keep the tensor core and the special-function units busy where one is a chain (B = 1, r = 16 over 6441 keys in one
// range 55.9 -> 45.4 us; B = 16, H = 16, D = 64, r = 100 over 680 keys 18.5 -> 17.1).  Both need a block; at two and three
// blocks they gain little but lose nothing.  In ranges the streams' meeting costs what they gain (r = 400 over 2921
// keys in two ranges 20.7 -> 21.1), so those stay one stream.
static bool dual_streams(int tiles_per_cta, int r, int L, int splits) {
  return (tiles_per_cta == 1 || r <= kQRows) && splits <= 1 && L > kKeys;
}

void attention_plan(int B_eff, int H, int r, int L, int num_sms, int *tiles_per_cta, int *kv_splits) {
  const int nkv = (L + kKeys - 1) / kKeys;
  const long long groups = static_cast<long long>(H) * B_eff;
  double best = 0.0;
  *tiles_per_cta = 2;
  *kv_splits = 1;
  for (int tiles = 2; tiles >= 1; --tiles) {
    if (tiles == 1 && r <= kQRows) continue;                  // the same launch
    const bool pair = tiles == 2 && r > kQRows;
    const long long units = (r + tiles * kQRows - 1) / (tiles * kQRows) * groups;
    const double t_block = pair ? 1.6 : 1.0, rows = (r < tiles * kQRows ? r : tiles * kQRows) / static_cast<double>(kQRows);
    for (int s = 1; s <= kMaxRanges; ++s) {
      const int per = (nkv + s - 1) / s;
      double cost;
      if (s == 1) {
        cost = 3.5 + static_cast<double>((units + num_sms - 1) / num_sms) * (per * (pair ? 1.6 : 0.85) + (pair ? 4.0 : 3.0));
      } else {
        if (per < 4 || (nkv + per - 1) / per != s || g_max_clusters[s] <= 0) continue;   // at least four key blocks a range
        const double waves = static_cast<double>((units + g_max_clusters[s] - 1) / g_max_clusters[s]);
        cost = waves * (2.5 + 0.75 * s + 3.4 * rows + per * t_block) + 4.0 * (waves - 1.0);
      }
      if (best == 0.0 || cost < best) { best = cost; *tiles_per_cta = tiles; *kv_splits = s; }
    }
  }
}

cudaError_t launch_attention(const CUtensorMap &tmQ, const CUtensorMap &tmK, const CUtensorMap &tmV,
                             const AttnArgs &a, int num_sms, cudaStream_t st) {
  if (a.r <= 0 || a.L <= 0) return cudaErrorInvalidValue;
  const bool dual = dual_streams(a.tiles_per_cta, a.r, a.L, a.kv_splits);
  if (a.D == 64) return dual ? launch_d<64, true>(tmQ, tmK, tmV, a, num_sms, st) : launch_d<64, false>(tmQ, tmK, tmV, a, num_sms, st);
  if (a.D == 128) return dual ? launch_d<128, true>(tmQ, tmK, tmV, a, num_sms, st) : launch_d<128, false>(tmQ, tmK, tmV, a, num_sms, st);
  return cudaErrorInvalidValue;
}

}  // namespace fvar
