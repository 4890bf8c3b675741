// Plain CUDA-core GEMM, C[M,N] (op)= A[M,K] * W[N,K]^T with fp32 accumulation.
// It is the arithmetic path of the fp32 configuration (exact fp32 FMA, no tensor-core rounding) and serves
// shapes the tensor-core kernel does not take (ragged N or K).
#include "engine_state.cuh"

namespace nz {

namespace {
constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4;

template <typename T, int EPI>
__global__ void __launch_bounds__(256) gemm_simt_kernel(GemmArgs a) {
  pdl_wait();
  pdl_launch();
  const int M = a.M_dev ? min(a.M, *a.M_dev) : a.M;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M) return;
  __shared__ float As[BK][BM + 4];
  __shared__ float Ws[BK][BN + 4];
  const T* A = reinterpret_cast<const T*>(a.A);
  const T* W = reinterpret_cast<const T*>(a.W);
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;          // 16 x 16 threads, each a 4 x 4 micro-tile
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  const int lr = tid >> 2, lc = (tid & 3) * 4;     // loader: row 0..63, k offset 0,4,8,12
  for (int k0 = 0; k0 < a.K; k0 += BK) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int k = k0 + lc + e;
      const int am = m0 + lr, wn = n0 + lr;
      As[lc + e][lr] = (am < M && k < a.K) ? to_f32(A[(long long)am * a.lda + k]) : 0.f;
      Ws[lc + e][lr] = (wn < a.N && k < a.K) ? to_f32(W[(long long)wn * a.ldw + k]) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float av[TM], wv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = As[k][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) wv[j] = Ws[k][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(av[i], wv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty * TM + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx * TN + j;
      if (n >= a.N) continue;
      const long long o = (long long)m * a.ldc + n;
      if (EPI == kEpiStoreAct) reinterpret_cast<T*>(a.C)[o] = from_f32<T>(acc[i][j]);
      else if (EPI == kEpiStoreF32) reinterpret_cast<float*>(a.C)[o] = acc[i][j];
      else if (EPI == kEpiAddF32) reinterpret_cast<float*>(a.C)[o] += acc[i][j];
      else if (EPI == kEpiBiasTanhF32) reinterpret_cast<float*>(a.C)[o] = tanhf(acc[i][j] + a.bias[n]);
    }
  }
}

// ---- few outputs: a thread per output, 16 x 16 of them per CTA, K in chunks of 128 fetched whole.  With a handful of rows
// the 64 x 64 tiles above are one or two CTAs, each a chain of a load and two barriers per 16 k (11 us at 40 x 64 x 256);
// here the chain is two rounds of loads and K fused multiply-adds.  Same order of summation (k ascending, one accumulator),
// so the same bits: which of the two runs may depend on the number of rows.
constexpr int SB = 16, SK = 128;

template <typename T>
__device__ __forceinline__ float4 load4(const T* row, int k, int K, bool vec) {      // row[k .. k + 3], zeros from K on
  if constexpr (sizeof(T) == 4) {
    if (vec && k + 4 <= K) return *reinterpret_cast<const float4*>(row + k);
  }
  float v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = k + e < K ? to_f32(row[k + e]) : 0.f;
  return make_float4(v[0], v[1], v[2], v[3]);
}

template <typename T, int EPI>
__global__ void __launch_bounds__(256) gemm_simt_small_kernel(GemmArgs a, bool vec) {
  __shared__ __align__(16) float As[SB][SK + 4], Ws[SB][SK + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * SB, n0 = blockIdx.x * SB;
  const int lr = tid >> 5, lc = (tid & 31) * 4;    // loader: rows lr and lr + 8, four consecutive k
  const T* W = reinterpret_cast<const T*>(a.W);
  float4 av[2], wv[2];
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) wv[j] = load4<T>(W + (long long)min(n0 + lr + 8 * j, a.N - 1) * a.ldw, k0 + lc, a.K, vec);
  };                                               // (rows beyond the edge: not stored)
  if (a.early) fetch_w(0);
  pdl_wait();
  pdl_launch();
  const int M = a.M_dev ? min(a.M, *a.M_dev) : a.M;
  if (m0 >= M) return;
  const T* A = reinterpret_cast<const T*>(a.A);
  auto fetch = [&](int k0, bool w) {
#pragma unroll
    for (int j = 0; j < 2; ++j) av[j] = load4<T>(A + (long long)min(m0 + lr + 8 * j, M - 1) * a.lda, k0 + lc, a.K, vec);
    if (w) fetch_w(k0);
  };
  fetch(0, !a.early);
  float acc = 0.f;
  const int m = m0 + ty, n = n0 + tx;
  const long long o = (long long)m * a.ldc + n;
  const bool valid = m < M && n < a.N;
  float extra = 0.f;                               // what the epilogue reads
  if (EPI == kEpiAddF32 && valid) extra = reinterpret_cast<const float*>(a.C)[o];
  if (EPI == kEpiBiasTanhF32 && valid) extra = a.bias[n];
  for (int k0 = 0; k0 < a.K; k0 += SK) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      *reinterpret_cast<float4*>(&As[lr + 8 * j][lc]) = av[j];
      *reinterpret_cast<float4*>(&Ws[lr + 8 * j][lc]) = wv[j];
    }
    __syncthreads();
    if (k0 + SK < a.K) fetch(k0 + SK, true);
    const int kc = min(SK, a.K - k0);
#pragma unroll 8
    for (int k = 0; k + 4 <= kc; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(&As[ty][k]), w = *reinterpret_cast<const float4*>(&Ws[tx][k]);
      acc = fmaf(x.x, w.x, acc); acc = fmaf(x.y, w.y, acc); acc = fmaf(x.z, w.z, acc); acc = fmaf(x.w, w.w, acc);
    }
    for (int k = kc & ~3; k < kc; ++k) acc = fmaf(As[ty][k], Ws[tx][k], acc);
    __syncthreads();
  }
  if (!valid) return;
  if (EPI == kEpiStoreAct) reinterpret_cast<T*>(a.C)[o] = from_f32<T>(acc);
  else if (EPI == kEpiStoreF32) reinterpret_cast<float*>(a.C)[o] = acc;
  else if (EPI == kEpiAddF32) reinterpret_cast<float*>(a.C)[o] = extra + acc;
  else if (EPI == kEpiBiasTanhF32) reinterpret_cast<float*>(a.C)[o] = tanhf(acc + extra);
}

// ---- the same tile with the element-wise kernels around a layer's product in it: the RMSNorm of its rows on the way in, rotary embedding
// and KV append, or SwiGLU, on the way out.  At a few rows of a narrow model a launch is 2 to 3 us whatever it does, and these were four
// of a layer's nine (tiny shape, 4 requests, natural drafts: 72 launches a decode).  Same arithmetic in the same order as the kernels
// apart.  A CTA adds its 16 rows' squares up for itself.  The 16 columns are two runs of 8 whose columns belong together (the halves of a
// rotary pair, gate and up), 8 lanes apart.  The weights (constant) are asked for before the launch's dependency is resolved.
enum RowsOut { kRowsStore = 0, kRowsRope = 1, kRowsSwiGLU = 2 };
struct RowsArgs { GemmArgs g; const float* gain; float eps; RopeAppendArgs r; };

template <int OUT>
__global__ void __launch_bounds__(256) norm_gemm_rows_kernel(RowsArgs ra) {
  __shared__ __align__(16) float As[SB][SK + 4], Ws[SB][SK + 4];
  const GemmArgs& a = ra.g;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const int m0 = blockIdx.y * SB;
  const int lr = tid >> 5, lc = lane * 4;          // loader: rows lr and lr + 8 (a row is one warp's), four consecutive k
  // first columns of the two runs
  const int half = OUT == kRowsRope ? ra.r.hd >> 1 : 0, rot_cols = OUT == kRowsRope ? (ra.r.Hq + ra.r.Hkv) * ra.r.hd : 0;
  int n_lo = blockIdx.x * SB, n_hi = n_lo + 8, n_end = a.N;          // (columns beyond n_end + the run's offset: not stored)
  if (OUT == kRowsRope && n_lo < rot_cols) {
    const int h = n_lo / ra.r.hd, g = (n_lo - h * ra.r.hd) >> 4;
    n_lo = h * ra.r.hd + g * 8; n_hi = n_lo + half;
  }
  if (OUT == kRowsSwiGLU) { n_lo = blockIdx.x * 8; n_hi = n_lo + (a.N >> 1); n_end = a.N >> 1; }
  const float* W = reinterpret_cast<const float*>(a.W);
  float4 av[2], wv[2];
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) wv[j] = load4<float>(W + (long long)min((j ? n_hi : n_lo) + lr, a.N - 1) * a.ldw, k0 + lc, a.K, true);
  };
  fetch_w(0);
  pdl_wait();
  pdl_launch();
  const int M = a.M_dev ? min(a.M, *a.M_dev) : a.M;
  if (m0 >= M) return;
  const float* row[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) row[j] = reinterpret_cast<const float*>(a.A) + (long long)min(m0 + lr + 8 * j, M - 1) * a.lda;
  auto fetch_a = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) av[j] = load4<float>(row[j], k0 + lc, a.K, true);
  };
  // (what the epilogue reads, on its way meanwhile)
  const int m = m0 + ty, n = (tx < 8 ? n_lo : n_hi - 8) + tx;
  const bool valid = m < M && (tx < 8 ? n : n_lo + (tx - 8)) < n_end && n < a.N;
  float cs = 0.f, sn = 0.f;
  long long dst = -1;
  if constexpr (OUT == kRowsRope) {
    if (valid && n >= ra.r.Hq * ra.r.hd) dst = ra.r.kv_dst[m];
    if (valid && n < rot_cols) {
      const long long t = (long long)ra.r.tok_pos[m] * half + (n % ra.r.hd) % half;
      cs = ra.r.cos_tab[t]; sn = ra.r.sin_tab[t];
    }
  }
  fetch_a(0);
  float rs[2] = {0.f, 0.f};
  for (int k0 = 0; k0 < a.K; k0 += SK) {
    float4 v[2] = {av[0], av[1]};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (k0 > 0) v[j] = load4<float>(row[j], k0 + lc, a.K, true);
      if (k0 + lc < a.K) rs[j] += v[j].x * v[j].x + v[j].y * v[j].y + v[j].z * v[j].z + v[j].w * v[j].w;
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) rs[j] = rsqrtf(warp_sum(rs[j]) / (float)a.K + ra.eps);
  float acc = 0.f;
  for (int k0 = 0; k0 < a.K; k0 += SK) {
    const float4 gn = load4<float>(ra.gain, k0 + lc, a.K, true);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 x = av[j];
      *reinterpret_cast<float4*>(&As[lr + 8 * j][lc]) = make_float4(x.x * rs[j] * gn.x, x.y * rs[j] * gn.y, x.z * rs[j] * gn.z, x.w * rs[j] * gn.w);
      *reinterpret_cast<float4*>(&Ws[lr + 8 * j][lc]) = wv[j];
    }
    __syncthreads();
    if (k0 + SK < a.K) { fetch_a(k0 + SK); fetch_w(k0 + SK); }
    const int kc = min(SK, a.K - k0);              // (K is a multiple of 4 here)
#pragma unroll 8
    for (int k = 0; k < kc; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(&As[ty][k]), w = *reinterpret_cast<const float4*>(&Ws[tx][k]);
      acc = fmaf(x.x, w.x, acc); acc = fmaf(x.y, w.y, acc); acc = fmaf(x.z, w.z, acc); acc = fmaf(x.w, w.w, acc);
    }
    __syncthreads();
  }
  const float other = OUT == kRowsStore ? 0.f : __shfl_xor_sync(0xffffffffu, acc, 8);
  if (!valid) return;
  if (OUT == kRowsStore) {
    reinterpret_cast<float*>(a.C)[(long long)m * a.ldc + n] = acc;
  } else if (OUT == kRowsSwiGLU) {
    if (tx < 8) reinterpret_cast<float*>(a.C)[(long long)m * a.ldc + n] = acc / (1.f + __expf(-acc)) * other;
  } else {
    const float y = n >= rot_cols ? acc : tx < 8 ? acc * cs - other * sn : acc * cs + other * sn;
    const int q_cols = ra.r.Hq * ra.r.hd, h = n / ra.r.hd, c = n - h * ra.r.hd;
    if (n < q_cols) reinterpret_cast<float*>(a.C)[(long long)m * a.ldc + n] = y;
    else if (dst >= 0) {
      float* cache = reinterpret_cast<float*>(n < rot_cols ? ra.r.k_cache : ra.r.v_cache);
      cache[dst + (long long)(h - (n < rot_cols ? ra.r.Hq : ra.r.Hq + ra.r.Hkv)) * ra.r.kv_head_stride + c] = y;
    }
  }
}

// up to 96 large tiles: they would leave a third of the SMs idle and each SM one CTA's chain
inline bool few_tiles(int M, int N) { return (long long)((N + BN - 1) / BN) * ((M + BM - 1) / BM) <= 96; }

// ---- and with the draft head's gathers in it: A's rows are put together on the way in.  STATE: [s_l ; e_l] of Eq. 3, as in
// trans_gather_kernel (whose rows these are), C = tanh(acc + bias); else h_l + s_l of Eq. 2 (draft_x_kernel), C = acc.
template <bool STATE>
__global__ void __launch_bounds__(256) draft_gemm_rows_kernel(GemmArgs a, EngineState e, int l, const float* __restrict__ embed) {
  __shared__ __align__(16) float As[SB][SK + 4], Ws[SB][SK + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const int m0 = blockIdx.y * SB, n0 = blockIdx.x * SB;
  const int lr = tid >> 5, lc = lane * 4;          // loader: rows lr and lr + 8 (a row is one warp's), four consecutive k
  const float* W = reinterpret_cast<const float*>(a.W);
  float4 av[2], wv[2];
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) wv[j] = load4<float>(W + (long long)min(n0 + lr + 8 * j, a.N - 1) * a.ldw, k0 + lc, a.K, true);
  };
  fetch_w(0);
  pdl_wait();
  pdl_launch();
  const float *p0[2], *p1[2];                      // the row's two sources; null: zeros
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int bk = min(m0 + lr + 8 * j, a.M - 1), b = bk / e.Kmax, k = bk - b * e.Kmax;
    const float* h0 = e.h_f32 + (long long)b * (e.L + 1) * e.d;
    const long long lv = (long long)l * e.Bmax * e.Kmax;
    if (STATE) {
      const DraftSource src = draft_source(e, b, k, l);
      const bool live = src.code >= 0 && src.parent >= 0;
      p0[j] = !live ? nullptr : l == 1 ? h0 : e.state_lv + (lv + (long long)b * e.Kmax + src.parent) * e.d;
      p1[j] = !live ? nullptr : embed + (long long)(e.li.off[l - 1] + src.code) * e.d;
    } else {
      p0[j] = h0 + (long long)l * e.d;
      p1[j] = l == 1 ? h0 : e.state_lv + (lv + bk) * e.d;
    }
  }
  const float uh = e.draft_use_h ? 1.f : 0.f, us = e.draft_use_s ? 1.f : 0.f;
  auto fetch_a = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int k = k0 + lc;
      av[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k >= a.K) continue;
      if (STATE) {                                 // (d is a multiple of 4: four values come from one of the two)
        if (p0[j]) av[j] = *reinterpret_cast<const float4*>(k < e.d ? p0[j] + k : p1[j] + (k - e.d));
      } else {
        const float4 h = *reinterpret_cast<const float4*>(p0[j] + k), s = *reinterpret_cast<const float4*>(p1[j] + k);
        av[j] = make_float4(uh * h.x + us * s.x, uh * h.y + us * s.y, uh * h.z + us * s.z, uh * h.w + us * s.w);
      }
    }
  };
  fetch_a(0);
  const int m = m0 + ty, n = n0 + tx;
  const bool valid = m < a.M && n < a.N;
  const float bias = STATE && valid ? a.bias[n] : 0.f;
  float acc = 0.f;
  for (int k0 = 0; k0 < a.K; k0 += SK) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      *reinterpret_cast<float4*>(&As[lr + 8 * j][lc]) = av[j];
      *reinterpret_cast<float4*>(&Ws[lr + 8 * j][lc]) = wv[j];
    }
    __syncthreads();
    if (k0 + SK < a.K) { fetch_a(k0 + SK); fetch_w(k0 + SK); }
    const int kc = min(SK, a.K - k0);              // (a multiple of 4)
#pragma unroll 8
    for (int k = 0; k < kc; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(&As[ty][k]), w = *reinterpret_cast<const float4*>(&Ws[tx][k]);
      acc = fmaf(x.x, w.x, acc); acc = fmaf(x.y, w.y, acc); acc = fmaf(x.z, w.z, acc); acc = fmaf(x.w, w.w, acc);
    }
    __syncthreads();
  }
  if (valid) reinterpret_cast<float*>(a.C)[(long long)m * a.ldc + n] = STATE ? tanhf(acc + bias) : acc;
}

template <typename T>
void dispatch(const GemmArgs& a, cudaStream_t st) {
  const dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM);
  const bool small = few_tiles(a.M, a.N);
  const dim3 grid_s((a.N + SB - 1) / SB, (a.M + SB - 1) / SB);
  const bool vec = sizeof(T) == 4 && a.lda % 4 == 0 && a.ldw % 4 == 0 && ((uintptr_t)a.A & 15) == 0 && ((uintptr_t)a.W & 15) == 0;
  auto go = [&](auto large_kernel, auto small_kernel) {
    if (small) launch_pdl(small_kernel, grid_s, dim3(256), 0, st, a, vec);
    else launch_pdl(large_kernel, grid, dim3(256), 0, st, a);
  };
  switch (a.epilogue) {
    case kEpiStoreAct: go(gemm_simt_kernel<T, kEpiStoreAct>, gemm_simt_small_kernel<T, kEpiStoreAct>); break;
    case kEpiStoreF32: go(gemm_simt_kernel<T, kEpiStoreF32>, gemm_simt_small_kernel<T, kEpiStoreF32>); break;
    case kEpiAddF32: go(gemm_simt_kernel<T, kEpiAddF32>, gemm_simt_small_kernel<T, kEpiAddF32>); break;
    case kEpiBiasTanhF32: go(gemm_simt_kernel<T, kEpiBiasTanhF32>, gemm_simt_small_kernel<T, kEpiBiasTanhF32>); break;
    default: break;
  }
}
}  // namespace

// Narrow rows: every CTA of a product adds its rows' squares up, so the wider the row the more of that is done twice; and only where
// the product's own kernel would be the one of few outputs.  Two layers, four requests of 20 items, beam 5, apart -> inside, us (prompt /
// verified decode): d = 64 65 -> 49 / 172 -> 145, 128 100 -> 89 / 197 -> 167, 192 157 -> 126 / 244 -> 213, 256 216 -> 208 / 269 -> 237.  Beyond
// the line it would still gain, less of the call: 384 312 -> 304 / 350 -> 326, 512 425 -> 423 / 447 -> 415.
bool norm_gemm_rows_applies(int M, int N, int K, const void* A, long long lda, const void* W, const void* gain) {
  return K <= 256 && K % 4 == 0 && lda % 4 == 0 && few_tiles(M, N) && (((uintptr_t)A | (uintptr_t)W | (uintptr_t)gain) & 15) == 0;
}
void launch_norm_gemm_rows(const GemmArgs& a, const void* gain, float eps, const RopeAppendArgs* rope, bool swiglu, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return;
  LaunchScope ls(kcGemm, st);
  RowsArgs ra{};
  ra.g = a; ra.gain = (const float*)gain; ra.eps = eps;
  if (rope) ra.r = *rope;
  const dim3 grid(swiglu ? (a.N / 2 + 7) / 8 : (a.N + SB - 1) / SB, (a.M + SB - 1) / SB);
  launch_pdl(rope ? norm_gemm_rows_kernel<kRowsRope> : swiglu ? norm_gemm_rows_kernel<kRowsSwiGLU> : norm_gemm_rows_kernel<kRowsStore>, grid,
             dim3(256), 0, st, ra);
}

// fp32, where the product's own kernel would be the one of few outputs.
bool draft_gemm_rows_applies(int M, int N, const EngineState& e, const void* W) {
  return e.d % 4 == 0 && few_tiles(M, N) && ((uintptr_t)W & 15) == 0;
}
// a: C, ldc, W, ldw, M (= requests * Kmax), N, K (= d, or 2 d with `state`) and the bias of Eq. 3
void launch_draft_gemm_rows(const GemmArgs& a, const EngineState& e, int l, const void* embed, bool state, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return;
  LaunchScope ls(kcGemm, st);
  launch_pdl(state ? draft_gemm_rows_kernel<true> : draft_gemm_rows_kernel<false>, dim3((a.N + SB - 1) / SB, (a.M + SB - 1) / SB), dim3(256), 0, st,
             a, e, l, (const float*)embed);
}

void launch_gemm_simt(const GemmArgs& a, bool bf16, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return;
  LaunchScope ls(kcGemm, st);
  if (bf16) dispatch<__nv_bfloat16>(a, st);
  else dispatch<float>(a, st);
}

}  // namespace nz
