// Weight-streaming GEMM for launches of few rows (at most 128, or a few row tiles of 128: gemm_skinny_applies):  C[M,N] (op)= A[M,K] * W[N,K]^T  with the operands' roles
// swapped on the tensor core.
//
// With a handful of rows the product is bound by reading W once from HBM.  The 128-row MMA operand is therefore a
// 128 x 64 tile of W (16 KB per copy, the unit that has to be kept in flight), the rows of A are the MMA's N (MT = 32, 48, 64
// or 128), and the accumulator in TMEM is a 128 x MT block of C^T.  An output tile is 128 columns of C; the K range of a
// tile is split over the CTAs of a thread-block cluster (up to 8) so that every SM streams a share of W, whatever N.
// Pieces of the tile are dealt out to the cluster's warps, which add the parts in rank order -- the bits never depend on
// timing -- and run the same fused epilogue as the other tensor-core kernels.  Up to 48 rows every CTA sends its parts straight from
// its accumulator to the shared memory of the warps that add them (st.async on their mbarriers); beyond, where there is no room for
// them beside the ring, it leaves its block in its own, and the warps read their peers' behind a cluster barrier.  The barrier, the
// round trip of the reads and a second barrier before a CTA may leave are a launch's last 1.3 us: one request on the 16-layer d = 2048
// backbone, prompt of 40 rows / verified decode (20 rows a pass) 676 -> 635 / 1,344 -> 1,278 us without them.  (The 48-row accumulator
// alone, read / sent: prompt of 41 rows and drafts 779 / 702 us, prompt of five and passes of 45 rows 2,636 / 2,526.)
// A CTA issues the weight copies of its first ring round BEFORE the launch's dependency on the preceding kernel is
// resolved (W is constant data), and the kernel is sized for two CTAs per SM, so the weight stream of a launch starts
// while its predecessor is still draining.
// Every mbarrier wait is bounded, as in the other kernels.
#include <stdlib.h>

#include "gemm_epilogue.cuh"

namespace nz {

namespace {

using namespace gemm_detail;

template <int MT, bool PUSH> struct SkinnyCfg {
  static constexpr int kTileBytesW = 128 * BK * 2;
  static constexpr int kTileBytesX = MT * BK * 2;
  static constexpr int kStageBytes = kTileBytesW + kTileBytesX;
  // The parts of a split tile are sent to the shared memory of the CTAs that add them up (PUSH: up to 48 rows, where the room for
  // them leaves a ring of four), or left in the CTA's own for its peers to read.
  static constexpr int kStages = MT == 128 ? 3 : 4;
  static constexpr int kRecvParts = PUSH ? (MT == 32 ? 36 : 48) : 0;         // of 512 bytes
  static constexpr int kRecvBytes = kRecvParts * 512;
  static constexpr int kBarBytes = 192;
  // (the array is declared 1024-byte aligned; the kernel checks the slack that it really needs)
  static constexpr int kSlack = 512;
  // (an image of the accumulator reuses the ring: a CTA has one tile, and the ring is idle once it is accumulated)
  static constexpr int kSmemBytes = kStages * kStageBytes + kRecvBytes + kSlack + kBarBytes + MT * 4 /*row scales*/;
  static constexpr int kTmemCols = MT <= 32 ? 32 : MT <= 64 ? 64 : 128;
  // kind::f16 instruction descriptor: D = f32, A = B = bf16, both K-major, N = MT, M = 128.
  static constexpr uint32_t kInstrDesc =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MT >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  static_assert((MT + 31) / 32 * 32 * 512 <= kStages * kStageBytes, "the accumulator's image does not fit in the ring");
  static_assert(2 * (kSmemBytes + 1024) <= 228 * 1024, "two CTAs per SM");
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// 16 bytes to the shared memory of CTA `rank` of the cluster, at the address that `local` has in this CTA; they count towards the
// bytes that the mbarrier at `bar` (an address of this CTA's as well) of that CTA waits for.
__device__ __forceinline__ void st_peer_f4(uint32_t local, uint32_t bar, uint32_t rank, float x, float y, float z, float w) {
  uint32_t ra, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(bar), "r"(rank));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(ra), "f"(x), "f"(y), "f"(z), "f"(w), "r"(rb) : "memory");
}
// 16 bytes of the shared memory of CTA `rank` of the cluster, at the address that `local` has in this CTA.
__device__ __forceinline__ float4 ld_peer_f4(uint32_t local, uint32_t rank) {
  uint32_t ra;
  float4 v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ra) : "memory");
  return v;
}
// The first phase of a barrier that peers signal, waited for by a whole warp; bounded, and given up early when the CTA's abort flag
// (if given) is raised.  (All lanes ask, here and for the accumulator: with one lane asking for the others, what follows was compiled
// for a warp that may be split there, and the same prompt and decode took 730 / 1,393 us.)
__device__ __forceinline__ bool recv_wait(uint32_t bar, volatile uint32_t* abort_flag) {
  auto here = [&] {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar) : "memory");
    return __all_sync(0xffffffffu, ok != 0u);
  };
  if (here()) return true;
  const long long t0 = clock64();
  for (;;) {
    if (here()) return true;
    if (__any_sync(0xffffffffu, (abort_flag && *abort_flag) || clock64() - t0 > kWaitCycles)) return false;
  }
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[16]) {
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
template <int MT, bool PUSH, int EPI>
__global__ void __launch_bounds__(kSkinnyThreads, 2)
    gemm_skinny_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, GemmArgs a,
                       int splits, int* status) {
  using C = SkinnyCfg<MT, PUSH>;
  constexpr int STAGES = C::kStages;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  if (base - smem_u32(smem_raw) > (uint32_t)C::kSlack) {      // (of every CTA alike) less aligned than declared: report, touch nothing
    pdl_wait();
    if (threadIdx.x == 0) atomicOr(status, kStInternal);
    return;
  }
  uint8_t* gen_base = smem_raw + (base - smem_u32(smem_raw));
  constexpr int kRecvAt = STAGES * C::kStageBytes, kBarAt = kRecvAt + C::kRecvBytes;
  const uint32_t recv_base = base + kRecvAt, bar_base = base + kBarAt;
  // barriers: full[STAGES], empty[STAGES], acc_full, recv[epilogue warps]; then the TMEM slot and the abort flag; then the rows' norm scales
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
  const uint32_t acc_full = bar_base + 8u * (2 * STAGES);
  auto recv_bar = [&](int w) { return bar_base + 8u * (2 * STAGES + 1 + w); };      // the parts of epilogue warp w's units are here
  constexpr int kSlotAt = 8 * (2 * STAGES + 1 + kSkinnyEpiWarps);
  static_assert(kSlotAt + 8 <= C::kBarBytes, "barrier area");
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen_base + kBarAt + kSlotAt);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  float* row_scale = reinterpret_cast<float*>(gen_base + kBarAt + C::kBarBytes);

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
    for (int w = 0; w < kSkinnyEpiWarps; ++w) mbar_init(recv_bar(w), 1);
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
  if (PUSH) cluster_arrive_relaxed();             // this CTA's barriers may be signalled (waited for before the first signal)
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
  ChunkCtx cc;
  int pos = 0;
  long long kvd = -1;
  auto fetch = [&](int u) {
    const int n_chunk = n0 + 32 * (u / quads), r = 4 * (u % quads) + rsub;
    if (EPI == kEpiRopeKV && r < rows) { pos = a.f.tok_pos[m0 + r]; kvd = a.f.kv_dst[m0 + r]; }
    cc = chunk_ctx<EPI>(a, n_chunk, k8);
    if (r < rows) aux = epi_prefetch<EPI>(a, cc, m0 + r, n_chunk + 4 * k8, pos);
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
    if constexpr (PUSH) {
      // what this warp's units will be sent (nobody signals the barrier before the peers' barriers are known to exist)
      if (mine && lane == 0) mbar_expect_tx(recv_bar(ew), (uint32_t)((units - u_first + u_step - 1) / u_step * splits * 512));
      cluster_wait();
    }
    const bool ok = warp_wait_uniform(acc_full, 0, abort_flag);
    tc_fence_after();
    // TMEM lane = column n0 + 32 q + lane, TMEM column = row; the two warps of a lane quarter take turns at the rows.
    constexpr int kLd = MT >= 64 ? 16 : 8;
    const int q = warp & 3, half = ew >> 2;
    if constexpr (PUSH) {
      // A lane's four rows of a unit are 16 bytes, a unit's part is 512.  (Also after a wait that expired: the peers count on it.)
      if (q < col_groups) {
#pragma unroll 1
        for (int r0 = half * kLd; r0 < rows; r0 += 2 * kLd) {
          float v[kLd];
          tmem_ld(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)r0, v);
#pragma unroll
          for (int j = 0; j < kLd; j += 4) {
            const int u = q * quads + ((r0 + j) >> 2);
            if (r0 + j < rows) {
              const int slot = u / splits, owner = u - slot * splits;
              st_peer_f4(recv_base + (uint32_t)((slot * splits + split) * 512 + lane * 16), recv_bar(slot & (kSkinnyEpiWarps - 1)), (uint32_t)owner,
                         v[j], v[j + 1], v[j + 2], v[j + 3]);
            }
          }
        }
      }
    } else if (ok) {
      // The image of a 32 x 32 block is 32 lines of one row each, their 16-byte chunks swizzled by the row.
      float* img = reinterpret_cast<float*>(gen_base) + q * 1024;
#pragma unroll 1
      for (int r0 = half * kLd; r0 < rows; r0 += 2 * kLd) {
        float v[kLd];
        tmem_ld(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)r0, v);
        float* blk = img + (r0 >> 5) * 4096;
#pragma unroll
        for (int j = 0; j < kLd; ++j) {
          const int r = (r0 & 31) + j;
          blk[(r * 8 + ((lane >> 2) ^ (r & 7))) * 4 + (lane & 3)] = v[j];
        }
      }
    }
    if (!ok && lane == 0) *abort_flag = 1;       // (behind the collective loads, which want the warp's lanes together)
  }
  if constexpr (PUSH) {
    if (!live || warp < 2) cluster_wait();       // (the epilogue warps of a live tile have)
    cluster_arrive_relaxed();                    // this CTA's parts are on their way
    // The row scales are in place: a unit's are another warp's work, and no barrier of the whole block comes before they are read.
    // (Here, under the parts' way: behind the scales it cost five requests' decode 1,318 -> 1,349 us.)
    if (live && warp >= 2 && a.f.ss_in) asm volatile("barrier.sync.aligned 1, %0;" ::"n"(32 * kSkinnyEpiWarps) : "memory");
    if (mine && !recv_wait(recv_bar(ew), abort_flag)) *abort_flag = 1;
  } else {
    // All parts are in place behind this barrier (or their CTA has raised its abort flag).
    if (splits > 1) cluster_sync_all();
    else __syncthreads();
  }
  if (mine && !*abort_flag) {
    // ------------------------------------------------------------------ epilogue, second half: the parts of a unit, added in rank order
#pragma unroll 1
    for (int u = u_first; u < units; u += u_step) {
      const int g = u / quads, r = 4 * (u - g * quads) + rsub, n_chunk = n0 + 32 * g, row = m0 + r;
      float4 x;
      if constexpr (PUSH) {
        // added as they came (lane = column, four rows), then turned in the room of the first part: lane = row, four columns
        float4* part = reinterpret_cast<float4*>(gen_base + kRecvAt) + u / splits * splits * 32 + lane;
        x = part[0];
#pragma unroll
        for (int sp = 1; sp < 8; ++sp)
          if (sp < splits) {
            const float4 y = part[sp * 32];
            x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
          }
        __syncwarp();
        float* turn = reinterpret_cast<float*>(part - lane);
        turn[lane] = x.x; turn[32 + lane] = x.y; turn[64 + lane] = x.z; turn[96 + lane] = x.w;
        __syncwarp();
        x = reinterpret_cast<const float4*>(turn)[lane];
      } else {
        const uint32_t at = base + (uint32_t)(((r >> 5) * 4 + g) * 4096 + ((r & 31) * 8 + (k8 ^ (r & 7))) * 16);
        if (splits > 1) {
          float4 part[8];
#pragma unroll
          for (int sp = 0; sp < 8; ++sp)
            if (sp < splits) part[sp] = ld_peer_f4(at, (uint32_t)sp);
          x = part[0];
#pragma unroll
          for (int sp = 1; sp < 8; ++sp)
            if (sp < splits) { x.x += part[sp].x; x.y += part[sp].y; x.z += part[sp].z; x.w += part[sp].w; }
          // A peer may be gone once all have arrived below, so its parts have to be here by then.  A unit has a row, whose store the warp
          // makes with the sum in hand; but a row without a place in the cache is not stored, so there the warp uses the sum now.
          if constexpr (EPI == kEpiRopeKV) x.x = __shfl_sync(0xffffffffu, x.x, lane);
        } else {
          x = *reinterpret_cast<const float4*>(gen_base + (at - base));
        }
      }
      const float rs = a.f.ss_in ? row_scale[r] : 1.f;
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
  if (PUSH || splits > 1) {                      // no CTA leaves while a peer may still send to it, or read its part
    // (Relaxed: what was read has been used.  A release waits for the stores to memory too: prompt and accepted tree of six requests on the
    // d = 2048 backbone 1,936 -> 1,966 us.)
    if (!PUSH) cluster_arrive_relaxed();
    cluster_wait();
    if (PUSH && mine && *abort_flag) recv_wait(recv_bar(ew), nullptr);      // given up before: everything sent has to land first
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols));
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(status, kStInternal);
}

template <int MT, bool PUSH, int EPI>
void launch(const GemmArgs& a, int tiles, int splits, cudaStream_t st) {
  using C = SkinnyCfg<MT, PUSH>;
  CUtensorMap tw, tx;
  if (!tma_map_bf16(a.W, a.N, a.K, a.ldw, 128, &tw) || !tma_map_bf16(a.A, a.M, a.K, a.lda, MT, &tx)) {
    static const int flag = kStInternal;       // cannot happen for shapes gemm_tc_supported accepted; report, do not guess
    cudaMemcpyAsync(a.status, &flag, sizeof(int), cudaMemcpyHostToDevice, st);
    return;
  }
  static PerDeviceOnce configured;
  configured.run([] {
    cudaFuncSetAttribute(gemm_skinny_kernel<MT, PUSH, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  });
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(tiles * splits, (a.M + MT - 1) / MT); cfg.blockDim = dim3(kSkinnyThreads); cfg.dynamicSmemBytes = C::kSmemBytes; cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = splits; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = pdl_enabled() ? 2 : 1;
  cudaLaunchKernelEx(&cfg, gemm_skinny_kernel<MT, PUSH, EPI>, tw, tx, a, splits, a.status);
}

template <int MT, bool PUSH>
void launch_epi(const GemmArgs& a, int tiles, int splits, cudaStream_t st) {
  switch (a.epilogue) {
    case kEpiStoreAct: launch<MT, PUSH, kEpiStoreAct>(a, tiles, splits, st); break;
    case kEpiStoreF32: launch<MT, PUSH, kEpiStoreF32>(a, tiles, splits, st); break;
    case kEpiAddF32: launch<MT, PUSH, kEpiAddF32>(a, tiles, splits, st); break;
    case kEpiBiasTanhF32: launch<MT, PUSH, kEpiBiasTanhF32>(a, tiles, splits, st); break;
    case kEpiSwiGLU: launch<MT, PUSH, kEpiSwiGLU>(a, tiles, splits, st); break;
    case kEpiAddNorm: launch<MT, PUSH, kEpiAddNorm>(a, tiles, splits, st); break;
    case kEpiRopeKV: launch<MT, PUSH, kEpiRopeKV>(a, tiles, splits, st); break;
    default: break;
  }
}

template <int MT>
void launch_mt(const GemmArgs& a, int tiles, int splits, cudaStream_t st) {
  if constexpr (MT <= 48) {
    // a CTA's share of at most MT units, each in `splits` parts, has to fit (at 48 rows that of 5 and of 7 CTAs does not)
    if (splits > 1 && (MT + splits - 1) / splits * splits <= SkinnyCfg<MT, true>::kRecvParts) {
      launch_epi<MT, true>(a, tiles, splits, st);
      return;
    }
  }
  launch_epi<MT, false>(a, tiles, splits, st);
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
  else if (a.M <= 48) launch_mt<48>(a, tiles, splits, st);
  else if (a.M <= 64) launch_mt<64>(a, tiles, splits, st);
  else launch_mt<128>(a, tiles, splits, st);
}

}  // namespace nz
