// CUDA-core attention: each token attends to a prefix of its request's context KV cache plus a few extra
// KV rows (its own tuple's drafted codes).  One warp per (token, query head); the warp is split into 4 groups
// of 8 lanes, each group walks every 4th position with the head dimension spread over its 8 lanes, and the
// 4 partial softmax states are merged at the end.  Exact fp32 arithmetic: this is the attention of the
// fp32 configuration and of head sizes the tensor-core kernel does not take.
#include <math.h>

#include "common.cuh"

namespace nz {

namespace {

template <int V> struct Int { static constexpr int value = V; };

template <typename T, int HD>
__global__ void __launch_bounds__(128) attn_simt_kernel(AttnArgs a) {
  constexpr int DPL = HD / 8;
  // Positions of a group in flight: their K and V rows are all asked for at once, 64 registers of them.  (With 16 floats a position and a
  // group's four in flight, a context of 61 took four round trips to the L2 in a row, 5.2 us a launch.)
  constexpr int U = HD >= 128 ? 2 : 256 / HD;
  constexpr int UX = 2;                            // draft rows: at most kMaxLevels, over four groups
  static_assert(4 * UX >= kMaxLevels, "draft rows");
  pdl_wait();
  pdl_launch();
  const int m = a.M_dev ? min(a.M, *a.M_dev) : a.M;
  const long long w = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5);
  const int i = (int)(w / a.Hq), h = (int)(w % a.Hq);
  if (i >= m) return;
  const int lane = threadIdx.x & 31, pg = lane >> 3, sub = lane & 7;
  const int kvh = h / (a.Hq / a.Hkv);
  const T* qp = reinterpret_cast<const T*>(a.q) + (long long)i * a.q_stride + (long long)h * HD + sub * DPL;
  float qv[DPL], acc[DPL];
#pragma unroll
  for (int j = 0; j < DPL; ++j) { qv[j] = to_f32(qp[j]) * a.scale; acc[j] = 0.f; }
  float m_run = -INFINITY, l_run = 0.f;

  // N positions (k / v: their rows, null = none) into the running softmax of the lane's group
  auto visit = [&](auto count, const T* const* kp, const T* const* vp) {
    constexpr int N = decltype(count)::value;
    float kv[N][DPL], vv[N][DPL], s[N];
#pragma unroll
    for (int u = 0; u < N; ++u)
#pragma unroll
      for (int j = 0; j < DPL; ++j) {
        kv[u][j] = kp[u] ? to_f32(kp[u][j]) : 0.f;
        vv[u][j] = kp[u] ? to_f32(vp[u][j]) : 0.f;
      }
    float m_new = m_run;
    bool any = false;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      s[u] = 0.f;
#pragma unroll
      for (int j = 0; j < DPL; ++j) s[u] = fmaf(qv[j], kv[u][j], s[u]);
      s[u] += __shfl_xor_sync(0xffffffffu, s[u], 1);
      s[u] += __shfl_xor_sync(0xffffffffu, s[u], 2);
      s[u] += __shfl_xor_sync(0xffffffffu, s[u], 4);
      if (kp[u]) { m_new = fmaxf(m_new, s[u]); any = true; }
    }
    if (!any) return;                              // (the same in the group's 8 lanes; scores that are not numbers, or -inf, go on)
    const float corr = (m_run == -INFINITY) ? 0.f : expf(m_run - m_new);
    l_run *= corr;
#pragma unroll
    for (int j = 0; j < DPL; ++j) acc[j] *= corr;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const float pw = kp[u] ? expf(s[u] - m_new) : 0.f;
      l_run += pw;
#pragma unroll
      for (int j = 0; j < DPL; ++j) acc[j] = fmaf(pw, vv[u][j], acc[j]);
    }
    m_run = m_new;
  };

  const int ctx_len = a.tok_ctx_len[i];
  const long long base = (long long)a.tok_row[i] * a.ctx_row_stride + (long long)kvh * a.ctx_head_stride + sub * DPL;
  const T* kc = reinterpret_cast<const T*>(a.k_ctx) + base;
  const T* vc = reinterpret_cast<const T*>(a.v_ctx) + base;
  for (int p0 = 0; p0 < ctx_len; p0 += 4 * U) {
    const T *kp[U], *vp[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int p = p0 + 4 * u + pg;
      kp[u] = p < ctx_len ? kc + (long long)p * HD : nullptr;
      vp[u] = vc + (long long)p * HD;
    }
    visit(Int<U>{}, kp, vp);
  }
  if (a.n_ext_max > 0) {
    const T *kp[UX], *vp[UX];
#pragma unroll
    for (int u = 0; u < UX; ++u) {
      const int e = 4 * u + pg;
      const long long off = (e < a.n_ext_max) ? a.tok_ext[(long long)i * a.n_ext_max + e] : -1;
      const long long eo = off + (long long)kvh * a.ext_head_stride + sub * DPL;
      kp[u] = off >= 0 ? reinterpret_cast<const T*>(a.k_ext) + eo : nullptr;
      vp[u] = reinterpret_cast<const T*>(a.v_ext) + eo;
    }
    visit(Int<UX>{}, kp, vp);
  }
  // merge the 4 position groups
#pragma unroll
  for (int o = 8; o <= 16; o <<= 1) {
    const float m_o = __shfl_xor_sync(0xffffffffu, m_run, o);
    const float l_o = __shfl_xor_sync(0xffffffffu, l_run, o);
    const float m_new = fmaxf(m_run, m_o);
    const float c_s = (m_run == -INFINITY) ? 0.f : expf(m_run - m_new);
    const float c_o = (m_o == -INFINITY) ? 0.f : expf(m_o - m_new);
    l_run = l_run * c_s + l_o * c_o;
#pragma unroll
    for (int j = 0; j < DPL; ++j) {
      const float a_o = __shfl_xor_sync(0xffffffffu, acc[j], o);
      acc[j] = acc[j] * c_s + a_o * c_o;
    }
    m_run = m_new;
  }
  if (pg == 0) {
    T* op = reinterpret_cast<T*>(a.out) + (long long)i * a.out_stride + (long long)h * HD + sub * DPL;
    const float inv = 1.f / l_run;
#pragma unroll
    for (int j = 0; j < DPL; ++j) op[j] = from_f32<T>(acc[j] * inv);
  }
}

template <typename T>
void dispatch(const AttnArgs& a, cudaStream_t st) {
  const long long warps = (long long)a.M * a.Hq;
  const int wpb = 4;
  dim3 grid((unsigned)((warps + wpb - 1) / wpb));
  switch (a.hd) {
    case 16: launch_pdl(attn_simt_kernel<T, 16>, grid, dim3(wpb * 32), 0, st, a); break;
    case 32: launch_pdl(attn_simt_kernel<T, 32>, grid, dim3(wpb * 32), 0, st, a); break;
    case 64: launch_pdl(attn_simt_kernel<T, 64>, grid, dim3(wpb * 32), 0, st, a); break;
    case 128: launch_pdl(attn_simt_kernel<T, 128>, grid, dim3(wpb * 32), 0, st, a); break;
    default: break;
  }
}
}  // namespace

void launch_attention_simt(const AttnArgs& a, bool bf16, cudaStream_t st) {
  if (a.M <= 0) return;
  LaunchScope ls(kcAttention, st);
  if (bf16) dispatch<__nv_bfloat16>(a, st);
  else dispatch<float>(a, st);
}

}  // namespace nz
