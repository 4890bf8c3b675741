// Plain CUDA-core GEMM, C[M,N] (op)= A[M,K] * W[N,K]^T with fp32 accumulation.
// It is the arithmetic path of the fp32 configuration (exact fp32 FMA, no tensor-core rounding) and serves
// shapes the tensor-core kernel does not take (ragged N or K).
#include "common.cuh"

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
  pdl_wait();
  pdl_launch();
  const int M = a.M_dev ? min(a.M, *a.M_dev) : a.M;
  if (m0 >= M) return;
  const T* A = reinterpret_cast<const T*>(a.A);
  float4 av[2], wv[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int am = min(m0 + lr + 8 * j, M - 1), wn = min(n0 + lr + 8 * j, a.N - 1);     // (rows beyond the edge: not stored)
      av[j] = load4<T>(A + (long long)am * a.lda, k0 + lc, a.K, vec);
      wv[j] = load4<T>(W + (long long)wn * a.ldw, k0 + lc, a.K, vec);
    }
  };
  fetch(0);
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
    if (k0 + SK < a.K) fetch(k0 + SK);
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

template <typename T>
void dispatch(const GemmArgs& a, cudaStream_t st) {
  const dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM);
  // up to 96 large tiles: they would leave a third of the SMs idle and each SM one CTA's chain
  const bool small = (long long)grid.x * grid.y <= 96;
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

void launch_gemm_simt(const GemmArgs& a, bool bf16, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return;
  LaunchScope ls(kcGemm, st);
  if (bf16) dispatch<__nv_bfloat16>(a, st);
  else dispatch<float>(a, st);
}

}  // namespace nz
