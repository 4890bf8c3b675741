// Blackwell tensor-core GEMM:  C[M,N] (op)= A[M,K] * W[N,K]^T,  bf16 operands, fp32 accumulation in TMEM.
//
// Persistent kernel: each CTA walks the 128 x BN output tiles assigned to it (BN = 32 ... 256, chosen so that small
// problems still spread over the SMs and large ones use the widest tile).  Warp 0 streams 128x64 (A) and BNx64 (W)
// bf16 tiles into a shared-memory ring with TMA (128-byte swizzle; K-major on both sides, which is exactly how
// activations [tokens, features] and weights [out, in] are stored).  Warp 1 issues tcgen05.mma (M128 N=BN K16, four per
// stage) into one of TWO BN-column TMEM accumulators and releases ring slots with tcgen05.commit.  Warps 2-9 (two per
// TMEM lane quarter) read a finished accumulator back with tcgen05.ld, 32 columns at a time, transpose the 32 x 32
// block through shared memory so that a warp writes whole row segments, and apply the epilogue -- while the MMA warp
// is already filling the other accumulator with the next tile.  Besides plain stores the epilogue can finish the
// surrounding element-wise work of a transformer layer: the RMSNorm row scale of the A operand, SwiGLU, rotary
// embedding + KV-cache append, residual add + next layer's norm input (see GemmFuse).
// Where the caller vouches for it (GemmArgs::early) a CTA reads the row count and asks for its first tile's weights, a ring full,
// while the preceding kernel still runs: with few rows that chain, not the tensor core, is the launch.  A request of five
// histories on the d = 2048 backbone (455 rows, then 45 a pass): 3040 -> 2944 us.
// Every mbarrier wait is bounded: on expiry the CTA raises an abort flag that ends every role's loop, records an error
// in the status word, drains the copies it has in flight, frees its TMEM and returns.
#include <stdlib.h>

#include "gemm_epilogue.cuh"

namespace nz {

int sm_count() {                                  // of the current device
  static std::mutex mu;
  static int n[kMaxDevices] = {};
  std::lock_guard<std::mutex> g(mu);
  const int dev = current_device();
  if (n[dev] == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
    cudaGetLastError();
    n[dev] = v;
  }
  return n[dev];
}

namespace {

using namespace gemm_detail;

template <int BN> struct Cfg {
  static constexpr int kTileBytesB = BN * BK * 2;
  static constexpr int kStageBytes = kTileBytesA + kTileBytesB;
  // as many stages as fit beside the transpose tiles: short-M launches are bound by bytes in flight per CTA
  static constexpr int kStages = BN >= 192 ? 4 : BN == 160 ? 5 : BN == 128 ? 6 : 8;
  static constexpr int kSmemBytes =
      kStages * kStageBytes + 1024 /*alignment slack*/ + 256 /*barriers*/ + kTransposeBytes;
  // kind::f16 instruction descriptor: D = f32, A = B = bf16, both K-major, N = BN, M = 128.
  static constexpr uint32_t kInstrDesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
};


template <int BN, int EPI>
__global__ void __launch_bounds__(kThreads) gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA,
                                                           const __grid_constant__ CUtensorMap tmB, GemmArgs a, int* status) {
  using C = Cfg<BN>;
  // two accumulators, in a power-of-two number of TMEM columns
  constexpr int kAccCols = 2 * BN;
  constexpr int kTmemCols = kAccCols <= 32 ? 32 : kAccCols <= 64 ? 64 : kAccCols <= 128 ? 128 : kAccCols <= 256 ? 256 : 512;
  constexpr int kFirstEpiWarp = 2;
  constexpr int STAGES = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bar_base = base + STAGES * C::kStageBytes;
  // barriers: full[STAGES], empty[STAGES], acc_full[2], acc_empty[2]; then the TMEM slot and the abort flag
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  auto acc_full = [&](int b) { return bar_base + 8u * (2 * STAGES + b); };
  auto acc_empty = [&](int b) { return bar_base + 8u * (2 * STAGES + 2 + b); };
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot =
      reinterpret_cast<volatile uint32_t*>(gen_base + STAGES * C::kStageBytes + 8 * (2 * STAGES + 4));
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k_iters = a.K / BK;
  const int M_early = !a.early ? 0 : a.M_dev ? min(a.M, __ldcg(a.M_dev)) : a.M;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), kEpiWarps); }
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_map(&tmA);
    tma_prefetch_map(&tmB);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // a.early: the first tile's weights are asked for at once, up to a ring full; the rows follow behind the wait
  int ahead = 0;                               // k-steps of the first tile whose weights are on their way (warp 0's)
  if (a.early && warp == 0) {
    const int M = M_early;
    const int tiles_m = (M + BM - 1) / BM, tiles_n = (a.N + BN - 1) / BN;
    if ((int)blockIdx.x < tiles_m * tiles_n) {
      const uint32_t leader = elect_one();
      ahead = min(STAGES, k_iters);
      for (int k = 0; k < ahead; ++k) {
        mbar_expect_tx_if(full_bar(k), C::kStageBytes, leader);
        tma_load_2d_if(base + k * C::kStageBytes + kTileBytesA, &tmB, k * BK, (int)blockIdx.x / tiles_m * BN, full_bar(k), leader);
      }
    }
  }
  // everything above needed nothing of the preceding kernel; from here on its results are read
  pdl_wait();
  pdl_launch();
  const int M = a.early ? M_early : a.M_dev ? min(a.M, *a.M_dev) : a.M;
  const int tiles_m = (M + BM - 1) / BM, tiles_n = (a.N + BN - 1) / BN;
  const int n_tiles = tiles_m * tiles_n;     // a CTA without a tile falls through every role loop

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    const uint32_t leader = elect_one();
    int it = 0;                                  // k-iterations issued so far, over all tiles
    int s = 0;                                   // it % STAGES, and the parity of slot s's current round
    uint32_t round = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile % tiles_m) * BM, n0 = (tile / tiles_m) * BN;
      for (int k = 0; k < k_iters; ++k, ++it) {
        // (waiting for the parity before the first one succeeds at once on a fresh barrier: round 0 never waits)
        if (!warp_wait_uniform(empty_bar(s), round ^ 1u, abort_flag)) { ok = false; break; }
        const uint32_t fb = full_bar(s), dst = base + s * C::kStageBytes;
        if (it >= ahead) {
          mbar_expect_tx_if(fb, C::kStageBytes, leader);
          tma_load_2d_if(dst + kTileBytesA, &tmB, k * BK, n0, fb, leader);
        }
        tma_load_2d_if(dst, &tmA, k * BK, m0, fb, leader);
        if (++s == STAGES) { s = 0; round ^= 1u; }
      }
    }
    if (!ok && lane == 0) {                      // drain: wait (bounded) for the copies still in flight
      *abort_flag = 1;
      for (int j = max(0, it - STAGES); j < it; ++j) mbar_wait(full_bar(j % STAGES), (j / STAGES) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    const uint32_t leader = elect_one();
    int t_local = 0, s = 0;
    uint32_t round = 0;
    bool ok = true;
    // descriptors of slot 0; a slot further on adds its byte offset / 16 to the address field (shared memory
    // addresses stay below 2^18, so the 14-bit field never carries)
    const uint64_t da0 = smem_desc(base), db0 = smem_desc(base + kTileBytesA);
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++t_local) {
      const int b = t_local & 1;
      if (t_local >= 2 && !warp_wait_uniform(acc_empty(b), ((t_local >> 1) - 1) & 1, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint32_t tmem_acc = tmem_base + (uint32_t)(b * BN);
      for (int k = 0; k < k_iters; ++k) {
        if (!warp_wait_uniform(full_bar(s), round, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint64_t so = (uint64_t)(s * (C::kStageBytes >> 4));
        tc_mma_kstep(tmem_acc, da0 + so, db0 + so, C::kInstrDesc, k > 0 ? 1u : 0u, leader);
        tc_commit_if(empty_bar(s), leader);          // slot free once these MMAs have read it
        if (++s == STAGES) { s = 0; round ^= 1u; }
      }
      if (ok) tc_commit_if(acc_full(b), leader);     // the accumulator is complete
    }
    if (!ok && leader) *abort_flag = 1;
  } else {
    // ------------------------------------------------------------------ epilogue (the last 8 warps)
    const int q = warp & 3;                      // TMEM lane quarter this warp may access
    const int half = (warp - kFirstEpiWarp) >> 2;   // which half of the tile's 32-column groups this warp takes
    float4* stg4 = reinterpret_cast<float4*>(gen_base + STAGES * C::kStageBytes + 256) + (warp - kFirstEpiWarp) * (32 * 8);
    int t_local = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++t_local) {
      const int tn = tile / tiles_m;
      const int m0 = (tile % tiles_m) * BM, n0 = tn * BN;
      const int b = t_local & 1;
      const EpiRow er = epilogue_row<EPI>(a, m0 + q * 32 + lane, M);   // overlaps the main loop
      EpiFirst first;
      epilogue_first<BN, EPI>(a, q, half, lane, m0, n0, M, er, first);
      ok = warp_wait_uniform(acc_full(b), (t_local >> 1) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after();
      drain_accumulator<BN, EPI>(a, tmem_base + (uint32_t)(b * BN), q, half, lane, stg4, m0, n0, M, er, first);
      // this warp is done reading the accumulator: hand it back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty(b));
    }
    if (!ok && lane == 0) *abort_flag = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols));
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(status, kStInternal);
}

// ---------------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------------
template <int BN, int EPI>
void launch(const GemmArgs& a, cudaStream_t st) {
  CUtensorMap ta, tb;
  if (!tma_map_bf16(a.A, a.M, a.K, a.lda, BM, &ta) || !tma_map_bf16(a.W, a.N, a.K, a.ldw, BN, &tb)) {
    static const int flag = kStInternal;       // cannot happen for shapes gemm_tc_supported accepted; report, do not guess
    cudaMemcpyAsync(a.status, &flag, sizeof(int), cudaMemcpyHostToDevice, st);
    return;
  }
  static PerDeviceOnce configured;
  configured.run([] {
    cudaFuncSetAttribute(gemm_tc_kernel<BN, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN>::kSmemBytes);
  });
  const long long tiles = (long long)((a.M + BM - 1) / BM) * ((a.N + BN - 1) / BN);
  const int grid = (int)(tiles < sm_count() ? tiles : sm_count());
  launch_pdl(gemm_tc_kernel<BN, EPI>, dim3(grid), dim3(kThreads), Cfg<BN>::kSmemBytes, st, ta, tb, a, a.status);
}

template <int BN>
void launch_bn(const GemmArgs& a, cudaStream_t st) {
  switch (a.epilogue) {
    case kEpiStoreAct: launch<BN, kEpiStoreAct>(a, st); break;
    case kEpiStoreF32: launch<BN, kEpiStoreF32>(a, st); break;
    case kEpiAddF32: launch<BN, kEpiAddF32>(a, st); break;
    case kEpiBiasTanhF32: launch<BN, kEpiBiasTanhF32>(a, st); break;
    case kEpiSwiGLU: launch<BN, kEpiSwiGLU>(a, st); break;
    case kEpiAddNorm: launch<BN, kEpiAddNorm>(a, st); break;
    case kEpiRopeKV: launch<BN, kEpiRopeKV>(a, st); break;
    default: break;
  }
}

}  // namespace

// Tiling of a launch: 32 ... 256 = output-tile width of the single-CTA kernel, kPlanPairs = 256 x 256 tiles on CTA pairs.
// Cost model in ns: a launch's fixed part + waves of tiles over the SMs (over the SM pairs) times (k-steps x the step of that
// tile + the part of the epilogue that nothing hides).  The steps are fitted to 114 shapes measured under every plan (200 to
// 4096 rows, N 512 to 22016, K 512 to 11008): the plan it picks is 0.6 % behind the best of each on average, the table of
// relative wave costs it replaces was 6 % (4096 rows x 896 x 896 14.4 -> 10.8 us, 2048 x 8192 at 200 rows 28 -> 23).  The tiling
// never changes the order in which a product's K range is summed, so it may depend on the row count.
// Beyond the fitted rows the pairs are taken unless the model has them 30 % behind: there launches are long and run back to back
// at the power cap, where a pair's lighter shared-memory traffic is clock.  Whole prompt passes of the 24-layer d = 896
// backbone, by the model alone / with pairs at 10 % / at 30 %: 6.5 k rows 6.37 / 6.08 / 6.05 ms, 7.7 k 7.41 / 7.03 / 7.02,
// 9.6 k 9.46 / 9.40 / 8.83, 23 k 21.1 / 20.9 / 20.9.  From 1,024 rows on: decodes of 2.6 k rows 2 % faster or 1 % slower.
constexpr int kPlanPairs = 512;
int gemm_tc_plan(int M, int N, int K) {
  static const bool no_pairs = getenv("NEZHA_NO_CTA_PAIRS") != nullptr;
  static const int forced = getenv("NEZHA_GEMM_PLAN") ? atoi(getenv("NEZHA_GEMM_PLAN")) : 0;   // experiments: a width, 512 = pairs
  static const int widths[6] = {256, 192, 160, 128, 64, 32}, step_ns[6] = {335, 323, 248, 213, 160, 101};
  constexpr int kPairStepNs = 312, kFixedNs = 3400, kPairFixedNs = 5500, kTailNs = 100;
  if (forced == kPlanPairs && M >= 1 && N >= 256) return kPlanPairs;
  for (int w : widths)
    if (forced == w) return forced;
  const long long tiles_m = (M + BM - 1) / BM, k_iters = K / BK;
  long long best = -1; int plan = 32;
  for (int i = 0; i < 6; ++i) {
    const int bn = widths[i];
    if (bn > 32 && N < bn) continue;
    const long long tiles = tiles_m * ((N + bn - 1) / bn);
    const long long cost = kFixedNs + (tiles + sm_count() - 1) / sm_count() * (k_iters * step_ns[i] + kTailNs);
    if (best < 0 || cost < best) { best = cost; plan = bn; }
  }
  if (!no_pairs && M > BM && N >= 256) {
    const long long pairs = sm_count() / 2;
    const long long tiles = ((M + 2 * BM - 1) / (2 * BM)) * (long long)((N + 255) / 256);
    const long long cost = kPairFixedNs + (tiles + pairs - 1) / pairs * (k_iters * kPairStepNs + kTailNs);
    if (M > 4096 ? 10 * cost < 13 * best : cost < best) { best = cost; plan = kPlanPairs; }
  }
  return plan;
}

bool gemm_tc_supported(const GemmArgs& a) {
  if (!a.status || !tma_encode_fn()) return false;
  if (a.K % BK || a.N % 32 || a.M <= 0) return false;
  if ((a.lda * 2) % 16 || (a.ldw * 2) % 16 || ((uintptr_t)a.A & 15) || ((uintptr_t)a.W & 15)) return false;
  if (((uintptr_t)a.C & 15) || (a.ldc & 3)) return false;          // the epilogue stores 8- and 16-byte vectors
  if (a.epilogue == kEpiBiasTanhF32 && ((uintptr_t)a.bias & 15)) return false;
  return a.epilogue >= kEpiStoreAct && a.epilogue <= kEpiRopeKV;
}

void launch_gemm_tc_pair(const GemmArgs& a, int n_sm, cudaStream_t st);
bool gemm_skinny_applies(const GemmArgs& a, int n_sm);
void launch_gemm_skinny(const GemmArgs& a, int n_sm, cudaStream_t st);

void launch_gemm_tc(const GemmArgs& a, cudaStream_t st) {
  LaunchScope ls(kcGemm, st);
  if (gemm_skinny_applies(a, sm_count())) { launch_gemm_skinny(a, sm_count(), st); return; }
  const int m_plan = a.M_expected > 0 && a.M_expected < a.M ? a.M_expected : a.M;
  switch (gemm_tc_plan(m_plan, a.N, a.K)) {
    case kPlanPairs: launch_gemm_tc_pair(a, sm_count(), st); break;
    case 256: launch_bn<256>(a, st); break;
    case 192: launch_bn<192>(a, st); break;
    case 160: launch_bn<160>(a, st); break;
    case 128: launch_bn<128>(a, st); break;
    case 64: launch_bn<64>(a, st); break;
    default: launch_bn<32>(a, st); break;
  }
}

}  // namespace nz
