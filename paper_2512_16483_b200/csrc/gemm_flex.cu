// GEMM on CTA pairs with a free tile width along the rows, sm_100a: out[R][N] = A[R][K] * W[N][K]^T.
//
// The weights are the M side of the MMA -- a pair of CTAs owns 256 output features, 128 each -- and a chunk of the rows,
// any multiple of 16 up to 256, is the N side.  With the roles that way round the row count of a step, which is whatever
// rank or batch asks for, costs no padding to 256, and the chunk width is free to make the number of tiles match the 74
// pairs of the chip.
//
// What bounds it: the operands' way from L2 (12 - 15 TB/s over the chip) and the tensor pipe, 0.10 + 0.00077 * width us per
// 64 of K and wave; a launch adds 2 us of set-up and first operands and 0.019 * width us of the last tile's epilogue.
// Against the best of the pairs of 256 rows (us, rows x features x K, launched through the kernel-level entry, which
// requests no weights early): 400 x 6144 x 2048 16.6 -> 13.9 with 160 rows a tile, 72 tiles; 283 x 8192 x 2048 16.9 -> 13.9;
// 680 x 4096 x 1024 10.8 -> 10.3; 2704 x 1024 x 1024 10.6 -> 9.5; 2704 x 1024 x 4096 25.6 -> 20.8; full tiles are level.  Multiples of 16 and not of 32 only (410 rows as two of 208 instead of 224,
// or three of 144 instead of 160) are worth 1.2 % of such a step: 3455 -> 3414 us, 408 rows 4015 -> 3951.  Spreading the K range of a tile over a cluster of pairs was built and left out:
// its reduction costs 4 - 6 us, 400 x 2048 x 8192 took 22.5 us against 21.7 of 128 x 128 tiles split the same way.
//
// The epilogue takes 32 rows at a time; what lies past the tile's end in its last chunk is the next tile's and not stored.
//
// Roles per CTA: warp 0 feeds the stage ring with TMA (cta_group::2: the bytes of both CTAs are counted on the barrier of
// the pair's even CTA), warp 1 of the even CTA issues the MMAs into one of two TMEM accumulators, warps 2-9 drain the
// other one: 32 features x 32 rows at a time through a staging tile, so that the results leave row by row in whole
// segments.  Every wait is bounded; on expiry the CTA flags the status word, gives its copies time to land, joins the
// pair's final barrier and frees its TMEM.
#include "gemm_common.cuh"
#include "gemm_rows.cuh"

namespace fvar {

constexpr int kFlexThreads = 64 + 32 * kEpiWarps;
constexpr int kFlexRing = 180224;                         // bytes of operand stages per CTA (176 KiB)
constexpr int kFlexMaxStages = 11;
constexpr int kFlexStage = 32 * 132;                      // staging tile of a warp: 32 rows x (32 features + 1) fp32
constexpr int kFlexSmemBytes = 1024 /*alignment*/ + kFlexRing + 256 /*barriers*/ + kEpiWarps * kFlexStage;
constexpr int kFlexWAtom = kBlockM * kBlockK * 2;         // 128 weight rows x 64 K
static_assert(kFlexSmemBytes <= 227 * 1024 && kFlexSmemBytes > 116 * 1024, "one CTA per SM");

// PRE: chunks of a warp whose residual is held in registers ahead of their sums (EPI_RESID; see launch_gemm_flex).
template <int EPI, int PRE>
__global__ void __launch_bounds__(kFlexThreads, 1)
gemm_flex_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ GemmArgs p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t tmem_base_holder;
  __shared__ volatile int abort_flag;

  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bar_base = ring + kFlexRing;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };                          // even CTA: both CTAs' bytes
  auto empty_bar = [&](int s) { return bar_base + 8u * (kFlexMaxStages + s); };      // one per CTA, signalled by the MMA commit
  auto tfull_bar = [&](int a) { return bar_base + 8u * (2 * kFlexMaxStages + a); };  // one per CTA, signalled by the MMA commit
  auto tempty_bar = [&](int a) { return bar_base + 8u * (2 * kFlexMaxStages + 2 + a); };   // even CTA: both CTAs' epilogue threads

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wb = wait_budget(p.wait_cycles);
  const uint32_t half = cluster_ctarank();                                            // 0: the even CTA of the pair
  const int nb = p.fx_nb, nk = p.fx_nk, nstages = p.fx_stages;
  const int tiles_f = (p.N + 2 * kBlockM - 1) / (2 * kBlockM), chunks = (p.R + nb - 1) / nb;
  const int total = tiles_f * chunks;
  constexpr bool kPart = EPI == EPI_PARTIAL;
  const int range = kPart ? static_cast<int>(cluster_id_x()) / total : 0;            // kPart: one tile and K range a pair
  const int tile0 = static_cast<int>(cluster_id_x()) - range * total, tile_step = kPart ? total : static_cast<int>(cluster_nctaid_x());
  const uint32_t b_bytes = static_cast<uint32_t>(nb / 2) * (kBlockK * 2);            // this CTA's rows of one K block
  const uint32_t stage_bytes = nk * (kFlexWAtom + b_bytes);
  const int num_kb = (p.K + kBlockK - 1) / kBlockK;
  const int nst = (num_kb + nk - 1) / nk / (kPart ? p.splits : 1);                   // stages of a tile
  const int k0 = kPart ? range * nst * nk : 0;                                       // first K block

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < nstages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull_bar(a), 1);
      mbar_init(tempty_bar(a), 2 * 32 * kEpiWarps);
    }
    mbar_fence_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmW);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_holder), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                 // the peer's barriers are initialised before anything signals them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  const uint32_t full0 = mapa_shared(full_bar(0), 0);
  const int pre = p.w_early ? min(nstages, nst) : 0;
  if (threadIdx.x == 0) {
    // While the predecessor drains: the weights of the first stages, which wait for nothing but the barriers just
    // initialised.  A loop of its own -- a test per stage inside the producer's made it miss its pace (400 x 6144 x 2048
    // 13.0 -> 14.9 us) and hid that this gains (Infinity 40 with table 3698 -> 3665 us).
    const int row_w = (2 * (tile0 / chunks) + static_cast<int>(half)) * kBlockM;
    for (int i = 0; i < pre; ++i) {
      if (half == 0) mbar_expect_tx(full_bar(i), 2u * stage_bytes);
      if (nk > 1) tma_load_3d_pair(ring + i * stage_bytes, &tmW, full0 + 8u * i, 0, row_w, k0 + i * nk);
      else tma_load_2d_pair(ring + i * stage_bytes, &tmW, full0 + 8u * i, (k0 + i) * kBlockK, row_w);
    }
  }
  pdl_wait();
  pdl_launch_dependents();
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------------- TMA producer (both CTAs)
      const int row_a0 = (tile0 % chunks) * nb + static_cast<int>(half) * (nb / 2);
      for (int i = 0; i < pre; ++i) {
        const uint32_t sa = ring + i * stage_bytes + nk * kFlexWAtom;
        if (nk > 1) tma_load_3d_pair(sa, &tmA, full0 + 8u * i, 0, row_a0, k0 + i * nk);
        else tma_load_2d_pair(sa, &tmA, full0 + 8u * i, (k0 + i) * kBlockK, row_a0);
      }
      int stage = pre == nstages ? 0 : pre, first = pre;
      uint32_t phase = pre == nstages ? 1u : 0u;
      bool issued = pre > 0;
      for (int tile = tile0; ok && tile < total; tile += tile_step) {
        const int ft = tile / chunks, ch = tile - ft * chunks;
        const int row_w = (2 * ft + static_cast<int>(half)) * kBlockM, row_a = ch * nb + static_cast<int>(half) * (nb / 2);
        for (int i = first; i < nst; ++i) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, p.status, &abort_flag, wb)) { ok = false; break; }
          if (half == 0) mbar_expect_tx(full_bar(stage), 2u * stage_bytes);
          const uint32_t sa = ring + stage * stage_bytes, fb = full0 + 8u * stage;
          if (nk > 1) {              // K blocks past the end of K are zero-filled and not multiplied
            tma_load_3d_pair(sa, &tmW, fb, 0, row_w, k0 + i * nk);
            tma_load_3d_pair(sa + nk * kFlexWAtom, &tmA, fb, 0, row_a, k0 + i * nk);
          } else {
            tma_load_2d_pair(sa, &tmW, fb, (k0 + i) * kBlockK, row_w);
            tma_load_2d_pair(sa + kFlexWAtom, &tmA, fb, (k0 + i) * kBlockK, row_a);
          }
          issued = true;
          if (++stage == nstages) { stage = 0; phase ^= 1u; }
        }
        first = 0;
      }
      if (!ok && issued) {
        // The byte counts of this CTA's copies go to the even CTA's barriers, which cannot be polled from here in
        // general: give the copies in flight a fixed time to land before shared memory is reused or released.
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000ll) {}
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (half == 0) {
      // ---------------------------------------------------------------- MMA issuer (even CTA of the pair)
      const uint32_t leader = elect_one() ? 1u : 0u;
      const uint32_t idesc = umma_idesc_bf16(2 * kBlockM, nb);
      int stage = 0, it = 0;
      uint32_t phase = 0;
      for (int tile = tile0; ok && tile < total; tile += tile_step, ++it) {
        const int a = it & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(tempty_bar(a), ((it >> 1) & 1u) ^ 1u, p.status, &abort_flag, wb));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * 256;
        uint32_t acc = 0u;
        for (int i = 0; i < nst; ++i) {
          ok = __all_sync(0xffffffffu, mbar_wait(full_bar(stage), phase, p.status, &abort_flag, wb));
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = ring + stage * stage_bytes;
          uint64_t dw = smem_desc_sw128(sa), da = smem_desc_sw128(sa + nk * kFlexWAtom);
          const int kvalid = min(nk, num_kb - k0 - i * nk);
          for (int kk = 0; kk < kvalid; ++kk) {
#pragma unroll
            for (int k = 0; k < kBlockK / 16; ++k) {
              umma_bf16_pair_if(leader, d_tmem, dw + 2 * k, da + 2 * k, idesc, acc);
              acc = 1u;
            }
            dw += kFlexWAtom >> 4;
            da += b_bytes >> 4;
          }
          umma_commit_pair_if(leader, empty_bar(stage));       // frees this stage in both CTAs
          if (++stage == nstages) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair_if(leader, tfull_bar(a));     // accumulator ready in both CTAs
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int quad = warp & 3, cg = (warp - 2) >> 2;       // features [32 quad, + 32); alternate 32-row chunks
    const uint32_t ep_stage = bar_base + 256 + (warp - 2) * kFlexStage;
    const uint32_t tempty0 = mapa_shared(tempty_bar(0), 0);
    int it = 0;
    for (int tile = tile0; ok && tile < total; tile += tile_step, ++it) {
      const int ft = tile / chunks, ch = tile - ft * chunks;
      const int a = it & 1, n0 = (2 * ft + static_cast<int>(half)) * kBlockM + quad * 32;
      const int row0 = ch * nb, rows = min(nb, p.R - row0);
      RowsEpilogue<EPI> ep(p, n0, ep_stage, lane, range, row0 + rows);
      // EPI_RESID: what the first PRE chunks read besides their sums is requested while the main loop runs (with one tile
      // a CTA nothing else hides it), the later ones' PRE ahead
      typename RowsEpilogue<EPI>::Fetch fetch[PRE];
#pragma unroll
      for (int u = 0; u < PRE; ++u)
        if (n0 < p.N && (cg + u * kEpiColGroups) * 32 < rows) ep.prefetch(row0 + (cg + u * kEpiColGroups) * 32, fetch[u]);
      ok = __all_sync(0xffffffffu, mbar_wait(tfull_bar(a), (it >> 1) & 1u, p.status, &abort_flag, wb));
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + a * 256 + (static_cast<uint32_t>(quad * 32) << 16);
      if (n0 < p.N) {                                                          // N % 64 == 0: whole 32-feature groups
#pragma unroll 1
        for (int c0 = cg; c0 * 32 < rows; c0 += PRE * kEpiColGroups) {
#pragma unroll
          for (int u = 0; u < PRE; ++u) {
            const int c = c0 + u * kEpiColGroups, ahead = c + PRE * kEpiColGroups;
            if (c * 32 >= rows) continue;
            uint32_t acc[32];
            tmem_ld32(taddr + c * 32, acc);
            tmem_ld_wait();
            ep.chunk(acc, row0 + c * 32, fetch[u]);
            if (ahead * 32 < rows) ep.prefetch(row0 + ahead * 32, fetch[u]);
          }
        }
      }
      tc_fence_before();
      mbar_arrive_cluster(tempty0 + 8u * a);
    }
  }

  // Nobody leaves (and no TMEM is freed) while the peer may still signal this CTA's barriers or the
  // pair's MMAs may still write this CTA's TMEM.
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// ------------------------------------------------------------------------------------------------ host
template <int EPI, int PRE>
static cudaError_t flex_prepare_one() {
  static bool ready = false;
  if (ready) return cudaSuccess;
  const cudaError_t err = cudaFuncSetAttribute(gemm_flex_kernel<EPI, PRE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFlexSmemBytes);
  if (err == cudaSuccess) ready = true;
  return err;
}

cudaError_t gemm_flex_prepare() {
  cudaError_t e = flex_prepare_one<EPI_F32, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_BF16, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_GELU_BF16, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_QKV, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_PARTIAL, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_RESID, 1>();
  if (e == cudaSuccess) e = flex_prepare_one<EPI_RESID, 2>();
  return e;
}

bool gemm_flex_supported(int epi, int N, int K) { return epi != EPI_ARGMAX && N % 64 == 0 && K % 8 == 0; }

// Pipeline shape for a.fx_nb rows a tile: two K blocks a stage (one TMA instruction an operand) when K is whole blocks
// and four such stages fit.
void gemm_flex_shape(GemmArgs &a) {
  const int kb_bytes = kFlexWAtom + a.fx_nb / 2 * kBlockK * 2;
  a.fx_nk = (a.K % kBlockK == 0 && a.K >= 2 * kBlockK && 8 * kb_bytes <= kFlexRing) ? 2 : 1;
  const int stages = kFlexRing / (a.fx_nk * kb_bytes);
  a.fx_stages = stages > kFlexMaxStages ? kFlexMaxStages : stages;
}

// The reduction of a K split over CTAs costs a cluster barrier and a round of remote reads after the last MMA, and the
// 128 x 128 tiles of that form (gemm_skinny.cu) move twice the operands of 256 x 224.  The kernel that reads the rows next
// can add up the ranges instead: the LayerNorm of the next block (400 x 2048 x 8192 with its gate and residual 25.9 us in the
// chain of a step, now 17 and 1 in the LayerNorm), or after a group's last block, whose rows are scattered and split for a
// projection, a pass of its own (26 us, now 17 and 3).
// Taken where the ranges fill most of the pairs: three or four of them, 0.6 of the pairs at work, two to four chunks of rows,
// the fewest that hold them (more and smaller chunks would put more pairs to work; not measured).  A step with ranges in every
// block and without (us):
//   2048 columns, K = 8192, four ranges, 64 pairs: 257 rows 3659 and 3934, 400 rows 4061 and 4253, 512 rows 4344 and 4424;
//   600 and 768 rows, where two ranges are all that fit: 5085 and 5039, 5554 and 5533 -- not taken;
//   1920 columns, K = 7680: 340 rows (64 pairs) 2361 and 2548, 510 rows 3012 and 3153, 680 rows (three ranges, 72 pairs) 3350 and 3515;
//   1024 columns, K = 4096: 576 rows (48 pairs) 787 and 858, 640 rows 833 and 885, 680 rows 1021 and 1041, 850 rows (64 pairs) 1205
//   and 1215; 400 and 510 rows (32 pairs) 786 and 770, 950 and 925, 1020 rows (64 full chunks) 1244 and 1231 -- not taken.
// One chunk (up to 256 rows) gains nowhere: 200 rows of 2048 columns 3365 and 3278.
int gemm_partial_plan(int R, int N, int K, int max_clusters, int *rows_tile) {
  const int chunks = (R + 255) / 256, num_kb = K / kBlockK, tiles = (N + 2 * kBlockM - 1) / (2 * kBlockM) * chunks;
  if (chunks < 2 || chunks > 4 || N > 2048 || K < 4096 || K % kBlockK != 0 || !gemm_flex_supported(EPI_PARTIAL, N, K)) return 0;
  *rows_tile = ((R + chunks - 1) / chunks + 15) / 16 * 16;
  if (chunks == 4 && *rows_tile > 224) return 0;
  for (int s = kMaxParts; s >= 3; --s)
    if (num_kb % (2 * s) == 0 && tiles * s <= max_clusters) return 5 * tiles * s >= 3 * max_clusters ? s : 0;
  return 0;
}

template <int EPI, int PRE>
static cudaError_t flex_launch_one(const CUtensorMap &tmA, const CUtensorMap &tmW, const GemmArgs &a, int max_clusters, cudaStream_t st) {
  const cudaError_t err = flex_prepare_one<EPI, PRE>();
  if (err != cudaSuccess) return err;
  const long long tiles = static_cast<long long>((a.N + 2 * kBlockM - 1) / (2 * kBlockM)) * ((a.R + a.fx_nb - 1) / a.fx_nb) * (EPI == EPI_PARTIAL ? a.splits : 1);
  if (EPI == EPI_PARTIAL && (tiles > max_clusters || a.K % (kBlockK * a.fx_nk * a.splits) != 0)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * static_cast<unsigned>(tiles < max_clusters ? tiles : max_clusters));
  cfg.blockDim = dim3(kFlexThreads);
  cfg.dynamicSmemBytes = kFlexSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = one_predecessor(st) ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_flex_kernel<EPI, PRE>, tmA, tmW, a);
}

// tmA: gemm_skinny_map over the activation rows (box of a.fx_nb / 2 rows), tmW: over the weight rows (box of 128), both
// with a.fx_nk K blocks.  max_clusters: resident CTA pairs (gemm_pair_max_clusters).
cudaError_t launch_gemm_flex(int epi, const CUtensorMap &tmA, const CUtensorMap &tmW, const GemmArgs &a, int max_clusters, cudaStream_t st) {
  if (a.nbatch != 1 || a.w_mn_major || (a.splits > 1 && epi != EPI_PARTIAL) || a.splits < 0 || a.R <= 0 || !gemm_flex_supported(epi, a.N, a.K) || a.fx_nb < 32 || a.fx_nb > 256 ||
      a.fx_nb % 16 || a.fx_stages < 2 || max_clusters <= 0)
    return cudaErrorInvalidValue;
  switch (epi) {
    case EPI_F32: return flex_launch_one<EPI_F32, 1>(tmA, tmW, a, max_clusters, st);
    case EPI_BF16: return flex_launch_one<EPI_BF16, 1>(tmA, tmW, a, max_clusters, st);
    case EPI_GELU_BF16: return flex_launch_one<EPI_GELU_BF16, 1>(tmA, tmW, a, max_clusters, st);
    case EPI_PARTIAL: return a.splits > 0 ? flex_launch_one<EPI_PARTIAL, 1>(tmA, tmW, a, max_clusters, st) : cudaErrorInvalidValue;
    case EPI_QKV: return flex_launch_one<EPI_QKV, 1>(tmA, tmW, a, max_clusters, st);
    // Up to 64 rows a tile each warp has one chunk, and the code for two only makes a cold launch longer: a step of 544 rows
    // of 2048 columns, where out-proj and cross out-proj take 64 rows a tile, 5001 against 5024 us (2364 rows of 1024
    // columns: level).  Beyond, two ahead is better than one (2704 rows, three scales: 5232 against 5272).
    case EPI_RESID:
      return a.fx_nb <= 64 ? flex_launch_one<EPI_RESID, 1>(tmA, tmW, a, max_clusters, st) : flex_launch_one<EPI_RESID, 2>(tmA, tmW, a, max_clusters, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace fvar
