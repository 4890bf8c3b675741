// Weight-streaming GEMM for launches of few rows (at most 128, or a few row tiles of 128: gemm_skinny_applies):  C[M,N] (op)= A[M,K] * W[N,K]^T  with the operands' roles
// swapped on the tensor core.
//
// With a handful of rows the product is bound by reading W once from HBM.  The 128-row MMA operand is therefore a
// 128 x 64 tile of W (16 KB per copy, the unit that has to be kept in flight), the rows of A are the MMA's N (MT = 32, 64
// or 128), and the accumulator in TMEM is a 128 x MT block of C^T.  An output tile is 128 columns of C; the K range of a
// tile is split over the CTAs of a thread-block cluster (up to 8) so that every SM streams a share of W, whatever N.
// Each CTA leaves its partial block in its own shared memory; after a cluster barrier pieces of the tile are dealt out to
// the cluster's warps, which add the parts in rank order, reading their peers' shared memory -- the bits never depend on
// timing -- and run the same fused epilogue as the other tensor-core kernels.
// A CTA issues the weight copies of its first ring round BEFORE the launch's dependency on the preceding kernel is
// resolved (W is constant data), and the kernel is sized for two CTAs per SM, so the weight stream of a launch starts
// while its predecessor is still draining.
// Every mbarrier wait is bounded, as in the other kernels.
#include <stdlib.h>

#include "gemm_epilogue.cuh"

namespace nz {

namespace {

using namespace gemm_detail;

template <int MT> struct SkinnyCfg {
  static constexpr int kTileBytesW = 128 * BK * 2;
  static constexpr int kTileBytesX = MT * BK * 2;
  static constexpr int kStageBytes = kTileBytesW + kTileBytesX;
  static constexpr int kStages = MT == 32 ? 5 : MT == 64 ? 4 : 3;
  static constexpr int kBarBytes = 128;
  // (the accumulator's image reuses the ring: a CTA has one tile, and the ring is idle once it is accumulated)
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + kBarBytes + MT * 4 /*row scales*/;
  static constexpr int kTmemCols = MT;
  // kind::f16 instruction descriptor: D = f32, A = B = bf16, both K-major, N = MT, M = 128.
  static constexpr uint32_t kInstrDesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  static_assert(MT * 512 <= kStages * kStageBytes, "the accumulator's image does not fit in the ring");
  static_assert(2 * (kSmemBytes + 1024) <= 228 * 1024, "two CTAs per SM");
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Every thread of every CTA of the cluster executes both halves, on every path.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 16 bytes of the shared memory of CTA `rank` of the cluster, at the address that `local` has in this CTA.
__device__ __forceinline__ float4 ld_peer_f4(uint32_t local, uint32_t rank) {
  uint32_t ra;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ra) : "memory");
  return v;
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

constexpr int kSkinnyEpiWarps = 8;
constexpr int kSkinnyThreads = 64 + 32 * kSkinnyEpiWarps;

// grid = (tiles x splits, row tiles), clusters of `splits` CTAs along x (blockIdx.x = tile * splits + split, split = rank in
// the cluster).  Warp 0: TMA producer; warp 1: TMEM owner and MMA issuer; warps 2 .. 9: epilogue.
// The epilogue is a chain of latencies behind the last MMA, so it is spread as thin as it goes: the tile's live rows are cut
// into units of 4 rows x 32 columns (one float4 per lane) that are dealt out to all epilogue warps of the cluster; a unit is
// one round of peer loads, and what it needs from memory is fetched before the accumulator is ready.  (One warp per 32 x 32
// block, the blocks dealt out to the CTAs, each row's norm scale added up by one lane: per launch at 20 rows 11.8 instead of 9.1 us for
// the output and down projections of the d = 2048 backbone, 7.8 instead of 5.4 for QKV.)
template <int MT, int EPI>
__global__ void __launch_bounds__(kSkinnyThreads, 2)
    gemm_skinny_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, GemmArgs a,
                       int splits, int* status) {
  using C = SkinnyCfg<MT>;
  constexpr int STAGES = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t bar_base = base + STAGES * C::kStageBytes;
  // barriers: full[STAGES], empty[STAGES], acc_full; then the TMEM slot and the abort flag; then the rows' norm scales
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  const uint32_t acc_full = bar_base + 8u * (2 * STAGES);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen_base + STAGES * C::kStageBytes + 8 * (2 * STAGES + 1));
  volatile uint32_t* abort_flag = tmem_slot + 1;
  float* row_scale = reinterpret_cast<float*>(gen_base + STAGES * C::kStageBytes + C::kBarBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x / splits, split = (int)cluster_rank();
  const int n0 = tile * 128, m0 = blockIdx.y * MT;
  // this CTA's share of the k-steps: contiguous, the first (k_iters % splits) shares one step longer
  const int k_iters = a.K / BK;
  const int k_base = k_iters / splits, k_rem = k_iters - k_base * splits;
  const int k_begin = split * k_base + min(split, k_rem), k_count = k_base + (split < k_rem ? 1 : 0);
  const int pre = min(STAGES, k_count);          // ring slots filled in the first round
  const int M_early = !a.early ? 0 : a.M_dev ? min(a.M, __ldcg(a.M_dev)) : a.M;
  const bool idle = a.early && M_early <= 0;      // a round queued for nothing: no row, and nothing is read (see k_run)
  // (a.early: one L2 latency less behind the wait, four times a layer; decode of one request, d = 2048: 2169 -> 2149 us)
  // the weight tiles of the first round are constant data, so they may be fetched while the predecessor still runs: for the first
  // row tile, which always goes through with its copies, and for the others where the rows are known already
  const bool w_ahead = (blockIdx.y == 0 && !idle) || m0 < M_early;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(acc_full, 1);
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_map(&tmW);
    tma_prefetch_map(&tmX);
    if (w_ahead)
      for (int s = 0; s < pre; ++s) {
        mbar_expect_tx(full_bar(s), C::kStageBytes);
        tma_load_2d(base + s * C::kStageBytes, &tmW, (k_begin + s) * BK, n0, full_bar(s));
      }
    // The down projection's next few k-steps into L2: the widest product by K behind the one that takes longest.  (4 steps, one
    // request drafted / verified: 821 -> 816 / 2148 -> 2134 us; 16 steps: nothing; the gate/up and QKV launches asking too: slower.)
    constexpr int kAhead = EPI == kEpiAddNorm ? 4 : 0;
    if (kAhead > 0 && w_ahead)
      for (int s = pre; s < min(k_count, pre + kAhead); ++s)
        asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(&tmW), "r"((k_begin + s) * BK), "r"(n0) : "memory");
    // behind them, in shares of 8 KB, the head of the next launch's weights (see kNextWeights in api.cu)
    if (blockIdx.y == 0 && !idle)
      for (long long o = (long long)blockIdx.x * 8192; o < a.next_w_bytes; o += (long long)gridDim.x * 8192) {
        const uint32_t bytes = (uint32_t)min(8192LL, a.next_w_bytes - o);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((const char*)a.next_w + o), "r"(bytes) : "memory");
      }
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)),
                 "r"(C::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  pdl_launch();
  const int M = a.early ? M_early : a.M_dev ? min(a.M, *a.M_dev) : a.M;
  const bool live = (blockIdx.y == 0 && !idle) || m0 < M;     // the same in all CTAs of a cluster
  // Without rows only the copies that are on their way are waited for (a surplus round of one request, 8 layers of d = 2048: 291 ->
  // 132 us).
  const int k_run = M > 0 ? k_count : pre;
  const int rows = max(0, min(MT, M - m0));       // rows of this tile that exist
  // units of the epilogue: unit u = columns n0 + 32 (u / quads) .., rows m0 + 4 (u % quads) ..
  const int ew = warp - 2, quads = (rows + 3) >> 2, col_groups = min(4, (a.N - n0) >> 5), units = col_groups * quads;
  const int u_step = splits * kSkinnyEpiWarps, u_first = split + splits * ew;     // (neighbouring units on different CTAs)
  const int k8 = lane & 7, rsub = lane >> 3;
  const bool mine = live && warp >= 2 && u_first < units;
  EpiAux aux;                                     // what the warp's next unit needs from memory
  int pos = 0;
  long long kvd = -1;
  auto fetch = [&](int u) {
    const int n_chunk = n0 + 32 * (u / quads), r = 4 * (u % quads) + rsub;
    if (EPI == kEpiRopeKV && r < rows) { pos = a.f.tok_pos[m0 + r]; kvd = a.f.kv_dst[m0 + r]; }
    if (r < rows) aux = epi_prefetch<EPI>(a, chunk_ctx<EPI>(a, n_chunk, k8), m0 + r, n_chunk + 4 * k8, pos);
  };

  if (!live) {
    // nothing to do for this row tile
  } else if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const uint32_t leader = elect_one();
    bool ok = true;
    int issued = pre;                            // k-steps whose `full` barrier has been armed
    for (int s = 0; s < pre; ++s) {
      if (!w_ahead) {
        mbar_expect_tx_if(full_bar(s), C::kStageBytes, leader);
        tma_load_2d_if(base + s * C::kStageBytes, &tmW, (k_begin + s) * BK, n0, full_bar(s), leader);
      }
      tma_load_2d_if(base + s * C::kStageBytes + C::kTileBytesW, &tmX, (k_begin + s) * BK, m0, full_bar(s), leader);
    }
    int s = 0;
    uint32_t round = 1;                          // parity bit of the round that k-step `pre` belongs to (pre = STAGES here)
    for (int k = pre; k < k_run; ++k, ++issued) {
      if (!warp_wait_uniform(empty_bar(s), round ^ 1u, abort_flag)) { ok = false; break; }
      const uint32_t fb = full_bar(s), dst = base + s * C::kStageBytes;
      mbar_expect_tx_if(fb, C::kStageBytes, leader);
      tma_load_2d_if(dst, &tmW, (k_begin + k) * BK, n0, fb, leader);
      tma_load_2d_if(dst + C::kTileBytesW, &tmX, (k_begin + k) * BK, m0, fb, leader);
      if (++s == STAGES) { s = 0; round ^= 1u; }
    }
    if (!ok && lane == 0) {                      // drain: wait (bounded) for the copies still in flight
      *abort_flag = 1;
      for (int j = max(0, issued - STAGES); j < issued; ++j) mbar_wait(full_bar(j % STAGES), (j / STAGES) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t leader = elect_one();
    bool ok = true;
    const uint64_t dw0 = smem_desc(base), dx0 = smem_desc(base + C::kTileBytesW);
    int s = 0;
    uint32_t round = 0;
    for (int k = 0; k < k_run; ++k) {
      if (!warp_wait_uniform(full_bar(s), round, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint64_t so = (uint64_t)(s * (C::kStageBytes >> 4));
      tc_mma_kstep(tmem_base, dw0 + so, dx0 + so, C::kInstrDesc, k > 0 ? 1u : 0u, leader);
      tc_commit_if(empty_bar(s), leader);
      if (++s == STAGES) { s = 0; round ^= 1u; }
    }
    if (ok) tc_commit_if(acc_full, leader);
    else if (leader) *abort_flag = 1;
  } else {
    // ------------------------------------------------------------------ epilogue, first half: the accumulator into shared memory
    // (under the main loop: the rows' norm scales, 8 lanes per row, each lane every eighth partial sum)
    for (int r = ew * 4 + rsub; r < ((rows + 3) & ~3); r += 4 * kSkinnyEpiWarps) {
      float ss = 0.f;
      if (a.f.ss_in && r < rows)
        for (int p = k8; p < a.f.ss_in_parts; p += 8) ss += a.f.ss_in[(long long)p * a.f.ss_ld + m0 + r];
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (k8 == 0) row_scale[r] = a.f.ss_in ? rsqrtf(ss * a.f.inv_dim + a.f.eps) : 1.f;
    }
    if (mine) fetch(u_first);
    const bool ok = warp_wait(acc_full, 0, abort_flag, lane);
    tc_fence_after();
    if (ok) {
      // TMEM lane = column n0 + 32 q + lane, TMEM column = row; each warp takes a half of the rows of its lane quarter.  The image
      // of a 32 x 32 block is 32 lines of one row each, their 16-byte chunks swizzled by the row.
      const int q = warp & 3, half = ew >> 2;
      float* img = reinterpret_cast<float*>(gen_base) + q * 1024;
#pragma unroll 1
      for (int r0 = half * (MT / 2); r0 < (half + 1) * (MT / 2) && r0 < rows; r0 += 16) {
        float v[16];
        tmem_ld16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)r0, v);
        float* blk = img + (r0 >> 5) * 4096;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int r = (r0 & 31) + j;
          blk[(r * 8 + ((lane >> 2) ^ (r & 7))) * 4 + (lane & 3)] = v[j];
        }
      }
    } else if (lane == 0) {
      *abort_flag = 1;
    }
  }
  // All parts are in place behind this barrier (or their CTA has raised its abort flag).
  if (splits > 1) cluster_sync_all();
  else __syncthreads();
  if (mine && !*abort_flag) {
    // ------------------------------------------------------------------ epilogue, second half: the parts of a unit, added in rank order
#pragma unroll 1
    for (int u = u_first; u < units; u += u_step) {
      const int g = u / quads, r = 4 * (u - g * quads) + rsub, n_chunk = n0 + 32 * g, row = m0 + r;
      const ChunkCtx cc = chunk_ctx<EPI>(a, n_chunk, k8);
      const uint32_t at = base + (uint32_t)(((r >> 5) * 4 + g) * 4096 + ((r & 31) * 8 + (k8 ^ (r & 7))) * 16);
      float4 x;
      if (splits > 1) {
        float4 part[8];
#pragma unroll
        for (int sp = 0; sp < 8; ++sp)
          if (sp < splits) part[sp] = ld_peer_f4(at, (uint32_t)sp);
        x = part[0];
#pragma unroll
        for (int sp = 1; sp < 8; ++sp)
          if (sp < splits) { x.x += part[sp].x; x.y += part[sp].y; x.z += part[sp].z; x.w += part[sp].w; }
      } else {
        x = *reinterpret_cast<const float4*>(gen_base + (at - base));
      }
      const float rs = row_scale[r];
      x = make_float4(x.x * rs, x.y * rs, x.z * rs, x.w * rs);
      const float4 back = epi_apply<EPI>(a, cc, r < rows, row, n_chunk + 4 * k8, k8, x, aux, kvd);
      if (EPI == kEpiAddNorm) {
        float ssq = back.x * back.x + back.y * back.y + back.z * back.z + back.w * back.w;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) ssq += __shfl_xor_sync(0xffffffffu, ssq, o);
        if (k8 == 0 && r < rows) a.f.ss_out[(long long)(n_chunk >> 5) * a.f.ss_ld + row] = ssq;
      }
      if (u + u_step < units) fetch(u + u_step);
    }
  }
  tc_fence_before();
  if (splits > 1) cluster_sync_all();            // no CTA leaves while a peer may still read its part
  else __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols));
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(status, kStInternal);
}

template <int MT, int EPI>
void launch(const GemmArgs& a, int tiles, int splits, cudaStream_t st) {
  using C = SkinnyCfg<MT>;
  CUtensorMap tw, tx;
  if (!tma_map_bf16(a.W, a.N, a.K, a.ldw, 128, &tw) || !tma_map_bf16(a.A, a.M, a.K, a.lda, MT, &tx)) {
    static const int flag = kStInternal;       // cannot happen for shapes gemm_tc_supported accepted; report, do not guess
    cudaMemcpyAsync(a.status, &flag, sizeof(int), cudaMemcpyHostToDevice, st);
    return;
  }
  static PerDeviceOnce configured;
  configured.run([] {
    cudaFuncSetAttribute(gemm_skinny_kernel<MT, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  });
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(tiles * splits, (a.M + MT - 1) / MT); cfg.blockDim = dim3(kSkinnyThreads); cfg.dynamicSmemBytes = C::kSmemBytes; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = splits; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = pdl_enabled() ? 2 : 1;
  cudaLaunchKernelEx(&cfg, gemm_skinny_kernel<MT, EPI>, tw, tx, a, splits, a.status);
}

template <int MT>
void launch_mt(const GemmArgs& a, int tiles, int splits, cudaStream_t st) {
  switch (a.epilogue) {
    case kEpiStoreAct: launch<MT, kEpiStoreAct>(a, tiles, splits, st); break;
    case kEpiStoreF32: launch<MT, kEpiStoreF32>(a, tiles, splits, st); break;
    case kEpiAddF32: launch<MT, kEpiAddF32>(a, tiles, splits, st); break;
    case kEpiBiasTanhF32: launch<MT, kEpiBiasTanhF32>(a, tiles, splits, st); break;
    case kEpiSwiGLU: launch<MT, kEpiSwiGLU>(a, tiles, splits, st); break;
    case kEpiAddNorm: launch<MT, kEpiAddNorm>(a, tiles, splits, st); break;
    case kEpiRopeKV: launch<MT, kEpiRopeKV>(a, tiles, splits, st); break;
    default: break;
  }
}

}  // namespace

// ---- which products of an engine run here, and how their K range is split.  Both are functions of N, K, the device and the
// engine's row class (the most rows a pass of it may have) only -- never of a launch's row count -- so a product's bits do not
// depend on its rows.
// Number of CTAs a tile's K range is split over (= the cluster size): as many as bring the grid of the class's row tiles to
// about two CTAs per SM (NEZHA_SKINNY_CTAS: another target), at most 8, each with at least four k-steps (64 KB of W per
// partial tile).  (One CTA per SM: 2.5 % more for a whole decode of the 16-layer d = 2048 backbone; its gate/up projection
// then has one CTA per tile.)
int gemm_skinny_splits(int N, int K, int row_class, int n_sm) {
  static const int forced = getenv("NEZHA_SKINNY_CTAS") ? atoi(getenv("NEZHA_SKINNY_CTAS")) : 0;
  const int target = forced > 0 ? forced : 2 * n_sm;
  const int tiles = (N + 127) / 128 * ((row_class + 127) / 128), k_iters = K / BK;
  int s = target / tiles;
  if (s > k_iters / 4) s = k_iters / 4;
  if (s > 8) s = 8;                              // the portable cluster size
  if (s < 1) s = 1;
  return s;
}

// Up to 128 rows every product is bound by reading W, and this kernel keeps more of it in flight.  With more rows W is
// shared by several row tiles and the general kernel's wider tiles win again -- except where its k-loop is the bound: one
// CTA walks all of K at 0.1 to 0.2 us per k-step, however few tiles there are, while here K is split.  One after another on cold
// weights, 256 / 384 / 512 / 640 rows, general -> this kernel, us: 2048 x 8192 24 -> 17 / 25 -> 27 / 25 -> 21 / 30 -> 25; 1536 x
// 8960 26 -> 17 / 25 -> 26 / 27 -> 28 / 27 -> 22; 896 x 4864 15 -> 9 / 16 -> 13 / 16 -> 13 / 16 -> 20; 2048 x 2048 9 -> 11 / 9 ->
// 17 / ..; 16384 x 2048 20 -> 21 / 27 -> 36 / ..; 6144 x 4096 19 -> 28 / 19 -> 22 / ..  The rule takes the first at 256 rows, the
// second to 384, the third at all four: the model of one class, not the best of each.
bool gemm_skinny_applies(const GemmArgs& a, int n_sm) {
  if (!a.skinny || a.M > a.skinny || a.skinny > kSkinnyClassRows) return false;
  if (a.skinny <= kSkinnyRows) return true;
  const int tiles = (a.N + 127) / 128 * ((a.skinny + 127) / 128), k_iters = a.K / BK;
  const int s = gemm_skinny_splits(a.N, a.K, a.skinny, n_sm);
  const int waves = (tiles * s + 2 * n_sm - 1) / (2 * n_sm), k_cta = (k_iters + s - 1) / s;
  const double here = waves * (7.0 + 0.75 * k_cta);
  const double there = 4.0 + 0.16 * k_iters;      // (its least: one wave of tiles)
  return here < 0.9 * there;
}

void launch_gemm_skinny(const GemmArgs& a, int n_sm, cudaStream_t st) {
  const int tiles = (a.N + 127) / 128, splits = gemm_skinny_splits(a.N, a.K, a.skinny, n_sm);
  if (a.M <= 32) launch_mt<32>(a, tiles, splits, st);      // (the bound, not the expected count: no row may be dropped)
  else if (a.M <= 64) launch_mt<64>(a, tiles, splits, st);
  else launch_mt<128>(a, tiles, splits, st);
}

}  // namespace nz
