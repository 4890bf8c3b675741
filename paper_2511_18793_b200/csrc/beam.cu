// Beam-search kernels: fused log-softmax + validity mask + beam top-k (one level of Algorithm 1 / Algorithm 3),
// the draft head's glue (Eq. 1-3 inputs), the verify pass's token list, and accept / roll-back (Algorithm 2's
// rejection and update steps).  Every kernel here runs one thread block per request; requests never interact.
#include <math.h>

#include "engine_state.cuh"

namespace nz {

// ====================================================================================================
// fused log-softmax + mask + top-k
// ====================================================================================================
// Per request: each warp takes beams r = warp, warp + n_warps, ...  For a beam it loads the T logits of the
// level's codebook (VPL per lane), computes log-softmax with warp shuffles, and extracts the beam's best
// candidates in order (repeated warp arg-max; ties to the smaller code):
//   per_beam <  T : the per_beam most probable codes, THEN the hash-set filter on those       (Algorithm 3: top-K, then verification)
//   per_beam >= T : the filter on all T codes, THEN the K best by cumulative log-probability  (top-k restricted to V)
// The sorted per-beam lists go to shared memory.  The K best of the request (ties to the smaller parent rank, then the smaller code) are
// ranked all with all among the candidates that the lists' order leaves in the running; more than kSelectKeys of those are merged
// list by list by warp 0.
namespace {

struct Cand { float s; int r; int t; };

__device__ __forceinline__ bool cand_better(float s, int r, int t, float s2, int r2, int t2) {
  if (s != s2) return s > s2;
  if (r != r2) return r < r2;
  return t < t2;
}

// Monotone map float -> unsigned (larger float, larger integer), so that a warp maximum is one redux instruction.
__device__ __forceinline__ unsigned ordered_bits(float f) {
  const unsigned u = __float_as_uint(f + 0.f);           // + 0: minus zero and plus zero rank alike
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(unsigned o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
constexpr unsigned kOrderedNegInf = 0x007fffffu;          // ordered_bits(-inf)

// Sorts v in descending order with Batcher's odd-even merge network (N a power of two; every index is a compile-time
// constant once unrolled, so v stays in registers).
template <int N>
__device__ __forceinline__ void sort_desc(unsigned long long (&v)[N]) {
#pragma unroll
  for (int p = 1; p < N; p <<= 1) {
#pragma unroll
    for (int k = p; k >= 1; k >>= 1) {
#pragma unroll
      for (int j = k % p; j + k < N; j += 2 * k) {
#pragma unroll
        for (int i = 0; i < k; ++i) {
          if (i + j + k < N && (i + j) / (2 * p) == (i + j + k) / (2 * p)) {
            const unsigned long long x = v[i + j], y = v[i + j + k];
            v[i + j] = x > y ? x : y;
            v[i + j + k] = x > y ? y : x;
          }
        }
      }
    }
  }
}

// One block per request.  Stage 1, a warp per input beam: log-softmax of the beam's logits row (+ Eq. 5 on every
// extension at the last level), then its `want` best codes in order into shared memory.  Stage 2: the K best of those
// lists (score, then parent rank, then code).  Stage 3, all threads: the output beams.  The kernel is a chain of
// dependent steps on a few warps, so its time is the sum of their latencies: loads whose address needs no other load
// go out together at the top; each lane keeps its keys sorted, so one survivor costs two redux and a shift; small
// merges are a rank count with no serial loop at all.
// Codebooks of more than 512 codes keep 32 keys per lane in registers besides the scores: that variant runs with at most
// 8 warps so that a thread may use up to 255 registers.
__host__ __device__ constexpr int select_max_threads(int vpl) { return vpl >= 32 ? 256 : 512; }
inline int select_warps(const SelectArgs& a) {
  const int cap = a.T > 512 ? 8 : 16;
  return a.in_stride < 8 ? 8 : a.in_stride > cap ? cap : a.in_stride;
}

// Candidates that the last stage compares all with all; more are merged list by list.
constexpr int kSelectKeys = 1024;
__host__ __device__ inline int select_keys(int in_stride, int K) { return ((in_stride * K < kSelectKeys ? in_stride * K : kSelectKeys) + 1) / 2 * 2; }

// Eq. 5 on the extensions of a beam that a lane answers for (codes lane, lane + 32, ...), 8 probes in flight: bit j = code
// lane + 32 j continues the prefix to a valid ID.
template <bool NARROW, int VPL>
__device__ __forceinline__ unsigned probe_extensions(unsigned long long* slots, unsigned long long n_buckets,
                                                  unsigned long long prefix_key, unsigned long long mult_n, int T) {
  const HashSetView hs{slots, n_buckets, NARROW};
  const int lane = threadIdx.x & 31;
  constexpr int PB = VPL < 8 ? VPL : 8;
  unsigned ok_mask = 0u;
#pragma unroll 1
  for (int j0 = 0; j0 < VPL; j0 += PB) {
    unsigned long long pk[PB]; bool want[PB], ok[PB];
#pragma unroll
    for (int j = 0; j < PB; ++j) {
      want[j] = lane + 32 * (j0 + j) < T;
      pk[j] = prefix_key + (unsigned long long)(lane + 32 * (j0 + j)) * mult_n;
    }
    hs_contains_form<NARROW, PB>(hs, pk, want, ok);
#pragma unroll
    for (int j = 0; j < PB; ++j) ok_mask |= (ok[j] ? 1u : 0u) << (j0 + j);
  }
  return ok_mask;
}

// PROBE: Eq. 5 on every extension of a beam by hash probes (select_probes).  A form of its own because the selection kernels
// are bound by instruction fetch and latency: the probes' straight-line code in all of them, where the default answers the
// mask from the prefix map, cost 1.4 % (16 layers, one request) to 3 % (4 layers, 64 requests) of a whole decode.
inline bool select_probes(const SelectArgs& a) { return a.filter && a.per_beam >= a.T && !a.prefix_filter && !a.final_mask_from_map; }

// What a fused kernel goes on with: the selection as it stands in shared memory (score, parent slot, code).
struct Selected { bool active; int gate, n; const float* s; const int* r; const int* t; };      // gate: the value that decided it
// 4 bytes of global memory into shared memory without passing through a register.
__device__ __forceinline__ void cp_async4(int* dst, const int* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_ints(int* dst, const int* src, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) cp_async4(dst + i, src + i);
}

// What differs from level to level.  (Apart from the kernel's parameters: a copy of those that a loop changes lives in local memory.)
struct SelectLevel {
  int n, T, per_beam, filter, prefix_filter, col_off, gate_value;
  const int* src_row; const int* in_codes; const float* in_score; const int* in_count;
  int* out_codes; float* out_score; int* out_parent; int* out_count;
};
__device__ __forceinline__ SelectLevel level_of(const SelectArgs& a) {
  return SelectLevel{a.n, a.T, a.per_beam, a.filter, a.prefix_filter, a.col_off, a.gate_value, a.src_row, a.in_codes, a.in_score, a.in_count,
                     a.out_codes, a.out_score, a.out_parent, a.out_count};
}

// s_codes: the input beams' codes in shared memory ([in_stride][tuple_len], brought by cp.async of all threads), or null.
template <int VPL, bool PROBE>
__device__ __forceinline__ Selected select_body(const SelectArgs& a, const SelectLevel& v, const int* s_codes = nullptr) {
  const int b = blockIdx.x;
  extern __shared__ unsigned char smem_raw[];
  const int nb_cap = a.in_stride;
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem_raw);      // [select_keys(nb_cap, K)] candidates in the running
  float* l_score = reinterpret_cast<float*>(s_key + select_keys(nb_cap, a.K));      // [nb_cap][K]
  int* l_tok = reinterpret_cast<int*>(l_score + (size_t)nb_cap * a.K);   // [nb_cap][K]
  int* l_cnt = l_tok + (size_t)nb_cap * a.K;                         // [nb_cap]
  float* sel_s = reinterpret_cast<float*>(l_cnt + nb_cap);           // [K] the selected (score, parent, code)
  int* sel_r = reinterpret_cast<int*>(sel_s + a.K);
  int* sel_t = sel_r + a.K;
  int* s_running = sel_t + a.K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;

  // ---- first wave of loads (none of these addresses depends on a loaded value)
  const int gate_v = a.gate_mode ? a.gate[b] : 0;
  const int nb_raw = v.in_count[b];
  const bool has0 = warp < nb_cap;                                   // this warp's first beam slot exists in the arrays
  const long long slot0 = (long long)b * a.in_stride + warp;
  const bool direct0 = has0 && !v.src_row && warp < a.src_mul;       // its logits row is known without a look-up
  long long row0 = 0;
  if (has0) row0 = v.src_row ? (long long)v.src_row[slot0] : (long long)b * a.src_mul + warp;
  const float base0 = has0 ? v.in_score[slot0] : 0.f;
  unsigned long long pk0 = 0;
  if (has0)
    for (int l = 0; l < v.n; ++l) pk0 += (unsigned long long)v.in_codes[slot0 * a.tuple_len + l] * a.li.mult[l];
  float bias[VPL], z0[VPL];
#pragma unroll
  for (int j = 0; j < VPL; ++j) {
    const int t = lane + 32 * j;
    bias[j] = (a.logit_bias && t < v.T) ? a.logit_bias[(long long)b * a.bias_stride + t] : 0.f;
    z0[j] = (direct0 && t < v.T) ? a.logits[row0 * a.row_stride + v.col_off + t] : 0.f;
  }
  if (a.gate_mode == 1 && gate_v != v.gate_value) return Selected{false, gate_v, 0, sel_s, sel_r, sel_t};
  if (a.gate_mode == 2 && !(gate_v < v.gate_value)) return Selected{false, gate_v, 0, sel_s, sel_r, sel_t};
  const int nb = min(nb_raw, nb_cap);
  if (threadIdx.x == 0) *s_running = 0;
  const bool all_codes = v.per_beam >= v.T;
  const int want = all_codes ? min(a.K, v.T) : min(v.per_beam, a.K);
  const unsigned long long mult_n = a.li.mult[v.n];

  for (int r = warp; r < nb; r += n_warps) {
    const bool first = r == warp;
    const long long slot = (long long)b * a.in_stride + r;
    const long long row = first ? row0 : (v.src_row ? (long long)v.src_row[slot] : (long long)b * a.src_mul + r);
    const float* z = a.logits + row * a.row_stride + v.col_off;
    float key[VPL];
    float mx = -INFINITY;
    if (!(first && direct0)) {       // (all under way before the first is used: one by one they took 2 to 4 us)
#pragma unroll
      for (int j = 0; j < VPL; ++j) z0[j] = lane + 32 * j < v.T ? z[lane + 32 * j] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      const int t = lane + 32 * j;
      key[j] = (t < v.T) ? z0[j] + bias[j] : -INFINITY;
      mx = fmaxf(mx, key[j]);
    }
    const float base = first ? base0 : v.in_score[slot];
    unsigned long long prefix_key = pk0;
    if (!first) {
      prefix_key = 0;
      for (int l = 0; l < v.n; ++l) prefix_key += (unsigned long long)v.in_codes[slot * a.tuple_len + l] * a.li.mult[l];
    }
    mx = warp_max(mx);
    float sum = 0.f;
#pragma unroll
    for (int j = 0; j < VPL; ++j) sum += (lane + 32 * j < v.T) ? expf(key[j] - mx) : 0.f;
    sum = warp_sum(sum);
    const float lse = mx + logf(sum);
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
      if (lane + 32 * j < v.T) {
        key[j] -= lse;                                   // log-probability
        if (all_codes) key[j] += base;                   // rank by cumulative log-probability
      }
    }
    // The bit set of the codes that may follow this beam: Eq. 5 for all T_L extensions at the last level, "some valid ID
    // begins with it" at an earlier level.
    const bool use_bits = v.prefix_filter || (all_codes && v.filter && a.final_mask_from_map);
    const unsigned long long* bits = use_bits ? pm_find(a.pm, v.n, prefix_key) : nullptr;
    if (all_codes && use_bits) {
#pragma unroll
      for (int j = 0; j < VPL; ++j) {
        const int t = lane + 32 * j;
        if (t < v.T && !pm_test(bits, t)) key[j] = -INFINITY;
      }
    } else if (PROBE && all_codes && v.filter) {
      const unsigned ok = a.hs.narrow ? probe_extensions<true, VPL>(a.hs.slots, a.hs.n_buckets, prefix_key, mult_n, v.T)
                                      : probe_extensions<false, VPL>(a.hs.slots, a.hs.n_buckets, prefix_key, mult_n, v.T);
#pragma unroll
      for (int j = 0; j < VPL; ++j)
        if (!((ok >> j) & 1u)) key[j] = -INFINITY;
    }
    int cnt = 0;
    if constexpr (VPL >= 16) {
      // Wide codebooks: no per-lane sort.  A sorting network of 16 or 32 keys is kilobytes of straight-line code that a
      // warp runs once, and fetching it costs more than it saves (12.6 us per beam at T = 512 against 3.2 at T = 256;
      // 6 us with this loop).  With many survivors per beam (K = 50) the sorted lists below are the cheaper form.
      // Each round every lane finds its best remaining key (four independent scans, so the chain is VPL / 4 long), the
      // warp picks the best of those (ties go to the smaller code), and the owner retires it: a short loop body.
      unsigned ob[VPL];                                  // ordered score bits; 0 = used up
#pragma unroll
      for (int j = 0; j < VPL; ++j) ob[j] = ordered_bits(key[j]);
#pragma unroll 1
      for (int it = 0; it < want; ++it) {
        unsigned qo[4]; int qj[4];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
          qo[q4] = 0u; qj[q4] = q4 * (VPL / 4);
#pragma unroll
          for (int j = q4 * (VPL / 4); j < (q4 + 1) * (VPL / 4); ++j)
            if (ob[j] > qo[q4]) { qo[q4] = ob[j]; qj[q4] = j; }
        }
        unsigned ho = qo[0]; int hj = qj[0];
#pragma unroll
        for (int q4 = 1; q4 < 4; ++q4)
          if (qo[q4] > ho) { ho = qo[q4]; hj = qj[q4]; }     // strict: the smaller code wins a tie
        const int ht = lane + 32 * hj;
        const unsigned mo = __reduce_max_sync(0xffffffffu, ho);
        if (mo <= kOrderedNegInf) break;
        const int bt = (int)__reduce_min_sync(0xffffffffu, ho == mo ? (unsigned)ht : 0x7fffffffu);
        if ((bt & 31) == lane) {
#pragma unroll
          for (int j = 0; j < VPL; ++j)
            if (j == (bt >> 5)) ob[j] = 0u;
        }
        if (lane == 0) {
          const float bv = from_ordered_bits(mo);
          l_score[(size_t)r * a.K + cnt] = all_codes ? bv : base + bv;
          l_tok[(size_t)r * a.K + cnt] = bt;
        }
        ++cnt;
      }
    } else {
      // this lane's keys in descending order: (ordered score bits, then the smaller code first); 0 = used up
      unsigned long long sk[VPL];
#pragma unroll
      for (int j = 0; j < VPL; ++j) sk[j] = ((unsigned long long)ordered_bits(key[j]) << 32) | (unsigned)(VPL - 1 - j);
      sort_desc<VPL>(sk);
      // ordered extraction: the warp's best head (ties go to the smaller code), whose lane then shifts its list
      for (int it = 0; it < want; ++it) {
        const unsigned ho = (unsigned)(sk[0] >> 32);
        const int ht = lane + 32 * (VPL - 1 - (int)(unsigned)sk[0]);
        const unsigned mo = __reduce_max_sync(0xffffffffu, ho);
        if (mo <= kOrderedNegInf) break;
        const int bt = (int)__reduce_min_sync(0xffffffffu, ho == mo ? (unsigned)ht : 0x7fffffffu);
        if ((bt & 31) == lane) {
#pragma unroll
          for (int j = 0; j + 1 < VPL; ++j) sk[j] = sk[j + 1];
          sk[VPL - 1] = 0ull;
        }
        if (lane == 0) {
          const float bv = from_ordered_bits(mo);
          l_score[(size_t)r * a.K + cnt] = all_codes ? bv : base + bv;
          l_tok[(size_t)r * a.K + cnt] = bt;
        }
        ++cnt;
      }
    }
    __syncwarp();
    if (!all_codes && (v.filter || v.prefix_filter)) {   // filter the chosen codes, keep their order
      int kept = 0;
      for (int c0 = 0; c0 < cnt; c0 += 32) {
        const int c = c0 + lane;
        bool ok = false; float sv = 0.f; int t = 0;
        if (c < cnt) {
          sv = l_score[(size_t)r * a.K + c]; t = l_tok[(size_t)r * a.K + c];
          ok = v.prefix_filter ? pm_test(bits, t) : hs_contains_thread(a.hs, prefix_key + (unsigned long long)t * mult_n);
        }
        const unsigned m = __ballot_sync(0xffffffffu, ok);
        __syncwarp();
        if (ok) {
          const int dst = kept + __popc(m & ((1u << lane) - 1u));
          l_score[(size_t)r * a.K + dst] = sv; l_tok[(size_t)r * a.K + dst] = t;
        }
        kept += __popc(m);
        __syncwarp();
      }
      cnt = kept;
    }
    if (lane == 0) l_cnt[r] = cnt;
  }
  __syncthreads();

  // ---- stage 2: the K best candidates of the nb lists into sel_*[0 .. n_out)
  // A candidate as one integer, larger = better: score, then the smaller parent rank, then the smaller code.
  auto cand_key = [&](int r, int c) {
    return (unsigned long long)ordered_bits(l_score[(size_t)r * a.K + c]) << 32 | (0xffffffffu - ((unsigned)r << 16 | (unsigned)l_tok[(size_t)r * a.K + c]));
  };
  // A list's scores do not rise: if all lists have m = ceil(K / nb) entries, K candidates score no less than the worst of their m-th, and
  // what scores less is out.  (By the score alone: where per_beam < T a list is in the order of the beam's own log-probabilities, and
  // two of them whose sums with the beam's score are rounded to the same number may stand there with the larger code first.  Each warp
  // finds the bound for itself.)
  const int m = nb > 0 ? (a.K + nb - 1) / nb : 1;
  int n_cand = 0;
  unsigned bound = ~0u;
  for (int r = lane; r < nb; r += 32) {
    const int c = l_cnt[r];
    n_cand += c;
    bound = min(bound, c >= m ? ordered_bits(l_score[(size_t)r * a.K + m - 1]) : 0u);
  }
  n_cand = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_cand);
  bound = __reduce_min_sync(0xffffffffu, bound);
  const int n_out = min(n_cand, a.K), key_cap = select_keys(nb_cap, a.K);
  for (int i0 = warp * 32; i0 < nb * a.K; i0 += blockDim.x) {
    const int i = i0 + lane, r = i / a.K, c = i - r * a.K;
    unsigned long long k = 0;
    if (r < nb && c < l_cnt[r]) k = cand_key(r, c);
    const bool in = k != 0ull && (unsigned)(k >> 32) >= bound;
    const unsigned ins = __ballot_sync(0xffffffffu, in);
    int at = 0;
    if (lane == 0 && ins) at = atomicAdd(s_running, __popc(ins));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(ins & ((1u << lane) - 1u));
    if (in && at < key_cap) s_key[at] = k;
  }
  __syncthreads();
  const int running = *s_running;
  if (running <= key_cap) {
    // a candidate's output position is the number of those that beat it (no two are equal).  Seven in a hundred candidates stay in
    // the running at 10 beams of 256 codes; a scan of the sorted lists per candidate took 3.7 us at K = 10 and 8 us at K = 20.
    for (int i = threadIdx.x; i < running; i += blockDim.x) {
      const unsigned long long k = s_key[i];
      int rank = 0;
#pragma unroll 4
      for (int j = 0; j < running; ++j) rank += s_key[j] > k ? 1 : 0;
      if (rank < a.K) {
        const unsigned rt = 0xffffffffu - (unsigned)k;
        sel_s[rank] = from_ordered_bits((unsigned)(k >> 32)); sel_r[rank] = (int)(rt >> 16); sel_t[rank] = (int)(rt & 0xffffu);
      }
    }
  } else if (warp == 0) {
    constexpr int RPL = 4;                                 // lists per lane: in_stride <= 128
    int ptr[RPL];
#pragma unroll
    for (int q = 0; q < RPL; ++q) ptr[q] = 0;
    if (!all_codes) {                                      // the equal sums of a list by their codes (see the bound)
      for (int r = lane; r < nb; r += 32)
        for (int c = 1; c < l_cnt[r]; ++c)
          for (size_t i = (size_t)r * a.K + c; i > (size_t)r * a.K && l_score[i - 1] == l_score[i] && l_tok[i - 1] > l_tok[i]; --i) {
            const int t = l_tok[i]; l_tok[i] = l_tok[i - 1]; l_tok[i - 1] = t;
          }
      __syncwarp();
    }
    for (int k = 0; k < a.K; ++k) {
      float bs = -INFINITY; int br = 0x7fffffff, bt = 0x7fffffff;
#pragma unroll
      for (int q = 0; q < RPL; ++q) {
        const int r = lane + 32 * q;
        if (r < nb && ptr[q] < l_cnt[r]) {
          const float sv = l_score[(size_t)r * a.K + ptr[q]];
          const int t = l_tok[(size_t)r * a.K + ptr[q]];
          if (br == 0x7fffffff || cand_better(sv, r, t, bs, br, bt)) { bs = sv; br = r; bt = t; }
        }
      }
      // warp arg-best: maximum score, then the smallest (parent rank, code) among the lanes that hold it
      const unsigned bo = br == 0x7fffffff ? 0u : ordered_bits(bs);
      const unsigned mo = __reduce_max_sync(0xffffffffu, bo);
      if (mo == 0u) break;                                   // every list is exhausted
      const unsigned pick = __reduce_min_sync(0xffffffffu, bo == mo ? ((unsigned)br << 16 | (unsigned)bt) : 0xffffffffu);
      br = (int)(pick >> 16); bt = (int)(pick & 0xffffu);
#pragma unroll
      for (int q = 0; q < RPL; ++q)
        if (lane + 32 * q == br) ++ptr[q];
      if (lane == 0) { sel_s[k] = from_ordered_bits(mo); sel_r[k] = br; sel_t[k] = bt; }
    }
  }
  if (s_codes) asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // ---- stage 3: the output beams, all threads
  for (int k = threadIdx.x; k < a.K; k += blockDim.x) {
    const long long o = (long long)b * a.out_stride + k;
    const bool live = k < n_out;
    v.out_score[o] = live ? sel_s[k] : -INFINITY;
    if (v.out_parent) v.out_parent[o] = live ? sel_r[k] : -1;
    if (a.out_token) a.out_token[o] = live ? sel_t[k] : -1;
  }
  if (v.out_codes) {
    for (int i = threadIdx.x; i < a.K * a.tuple_len; i += blockDim.x) {
      const int k = i / a.tuple_len, l = i - k * a.tuple_len;
      int c = -1;
      if (k < n_out) {
        if (l < v.n) c = s_codes ? s_codes[sel_r[k] * a.tuple_len + l] : v.in_codes[((long long)b * a.in_stride + sel_r[k]) * a.tuple_len + l];
        else if (l == v.n) c = sel_t[k];
      }
      v.out_codes[((long long)b * a.out_stride + k) * a.tuple_len + l] = c;
    }
  }
  if (threadIdx.x == 0) v.out_count[b] = n_out;
  // (what the kernels before this one reported; the host looks when the stream is idle, so nothing waits for the bus here: 1.5 us)
  if (a.host_status && b == 0 && threadIdx.x < 4) a.host_status[threadIdx.x] = *(volatile int*)(a.status + threadIdx.x);
  return Selected{true, gate_v, n_out, sel_s, sel_r, sel_t};
}

// Codes per lane of a codebook of T codes, as a constant.
template <int V> struct Vpl { static constexpr int value = V; };
template <typename F> void with_vpl(int T, F&& f) {
  if (T <= 32) f(Vpl<1>{});
  else if (T <= 256) f(Vpl<8>{});
  else if (T <= 512) f(Vpl<16>{});
  else f(Vpl<32>{});
}

template <int VPL, bool PROBE>
__global__ void __launch_bounds__(select_max_threads(VPL)) select_kernel(SelectArgs a) {
  pdl_wait();
  pdl_launch();
  select_body<VPL, PROBE>(a, level_of(a));
}

}  // namespace

cudaError_t select_step_configure(int bytes);
size_t advance_smem_bytes(int Kmax, int L);

size_t select_smem_bytes(int in_stride, int K) {
  return ((size_t)select_keys(in_stride, K) * sizeof(unsigned long long) + (size_t)in_stride * K * (sizeof(float) + sizeof(int)) + (size_t)in_stride * sizeof(int) +
          (size_t)K * (sizeof(float) + 2 * sizeof(int)) + sizeof(int) + 15) / 16 * 16;
}

// The attribute belongs to the device, and several contexts may share one: it is only ever raised.
cudaError_t select_configure(int max_beam) {
  static int configured_bytes[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  int bytes = (int)(select_smem_bytes(max_beam, max_beam) + advance_smem_bytes(max_beam, kMaxLevels));
  if (bytes <= configured_bytes[dev]) return cudaSuccess;
  configured_bytes[dev] = bytes;
  cudaError_t e = cudaSuccess;
  auto set = [&](auto vpl) {
    constexpr int V = decltype(vpl)::value;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_kernel<V, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_kernel<V, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set(Vpl<1>{}); set(Vpl<8>{}); set(Vpl<16>{}); set(Vpl<32>{});
  if (e != cudaSuccess) return e;
  return select_step_configure(bytes);
}

void launch_select(const SelectArgs& a, cudaStream_t st) {
  if (a.batch <= 0) return;
  const size_t smem = select_smem_bytes(a.in_stride, a.K);
  LaunchScope ls(kcSelect, st);
  const int warps = select_warps(a);   // a warp per beam where that fits
  const dim3 block(32 * warps);
  with_vpl(a.T, [&](auto vpl) {
    constexpr int V = decltype(vpl)::value;
    launch_pdl(select_probes(a) ? select_kernel<V, true> : select_kernel<V, false>, dim3(a.batch), block, smem, st, a);
  });
}

// ====================================================================================================
// small state kernels
// ====================================================================================================
namespace {

__global__ void fill_i32_kernel(int* p, long long n, int v) {
  pdl_wait();
  pdl_launch();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    p[i] = v;
}

// Start of a decode call, one block per request: B_0 = { empty beam, score 0 }, nothing settled, and the fill values of the
// call's outputs (out_* and the trace's pointers may be null; their slots of rounds that do not run keep these values).
// from_scratch: round 1 drafts, from the empty beam (Algorithm 3's initialisation).
__global__ void __launch_bounds__(128) decode_begin_kernel(EngineState e, int batch, int K, int from_scratch, int* out_codes,
                                                           float* out_scores, int* out_count, nezha_trace tr) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x, L = e.L, R = e.L - 1;
  if (b == 0 && threadIdx.x == 0) { *e.draft_rows = batch * e.Kmax; *e.n_tokens = 0; }
  if (threadIdx.x == 0) {
    e.tb_count[0 * e.Bmax + b] = 1;
    e.tb_score[lvl_bk(e, 0, b, 0)] = 0.f;
    e.tb_parent[lvl_bk(e, 0, b, 0)] = -1;
    e.tb_src[lvl_bk(e, 0, b, 0)] = -1;
    e.row_m[b] = 0;
    e.row_cur[b] = 0;
    e.row_spec[b] = 1;
    e.row_m_start[b] = 0;
    e.d_m[b] = from_scratch ? 0 : L;
    if (out_count) out_count[b] = 0;
  }
  for (int l = threadIdx.x; l <= L; l += blockDim.x) e.dw_count[(long long)l * e.Bmax + b] = l == 0 && from_scratch ? 1 : 0;
  if (from_scratch)
    for (int k = threadIdx.x; k < e.Kmax; k += blockDim.x) {
      const long long s = lvl_bk(e, 0, b, k);
      e.dw_score[s] = k == 0 ? 0.f : -INFINITY;
      e.dw_parent[s] = k == 0 ? 0 : -1;
      for (int l = 0; l < L; ++l) e.dw_codes[s * L + l] = -1;
    }
  if (out_scores) for (int i = threadIdx.x; i < K; i += blockDim.x) out_scores[(long long)b * K + i] = -INFINITY;
  auto fill = [&](int* p, int slices, int per) {       // [slices][batch][per]
    if (!p) return;
    for (int r = 0; r < slices; ++r)
      for (int i = threadIdx.x; i < per; i += blockDim.x) p[((long long)r * batch + b) * per + i] = -1;
  };
  fill(out_codes, 1, K * L);
  fill(tr.drafts, R, K * L); fill(tr.n_draft, R, 1); fill(tr.accepted_len, R, K); fill(tr.level_reached, R, 1);
  fill(tr.tree_codes, R * L, K * L); fill(tr.tree_count, R * L, 1);
}

// Caller-supplied drafted tuples for the round (or none: n_draft == nullptr and drafts == nullptr -> an empty tree).
// The tree of the tuples is built level by level: level j holds their distinct j-prefixes in order of first appearance
// (tuples that share a prefix share its node), each with the slot of its parent.  One block of >= Kmax threads per request.
__global__ void draft_set_kernel(EngineState e, int batch, int K, const int* drafts, const int* n_draft) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x;
  if (b == 0 && threadIdx.x == 0) *e.n_tokens = 0;
  if (b >= batch) return;
  const int L = e.L, k = threadIdx.x;
  __shared__ int s_slot[2][128];                 // slot of tuple k's prefix in the previous / the current level
  __shared__ int s_new[128], s_ok[128], s_cnt;
  const int cnt = (drafts && e.row_m[b] < L) ? max(0, min(n_draft[b], K)) : 0;
  int code[kMaxLevels];
  bool ok = k < cnt;
  for (int l = 0; l < L; ++l) {
    code[l] = ok ? drafts[((long long)b * K + k) * L + l] : -1;
    if (k < cnt && (code[l] < 0 || code[l] >= e.li.T[l])) { atomicOr(e.status, kStBadCode); ok = false; }
  }
  s_slot[0][k] = 0;                              // level 0: the empty prefix, slot 0
  s_ok[k] = ok ? 1 : 0;                          // a tuple with an out-of-range code is dropped as a whole
  __syncthreads();
  for (int j = 1; j <= L; ++j) {
    const int cur = j & 1, prev = cur ^ 1;
    int first = -1;                              // the first tuple with the same j-prefix
    if (ok) {
      for (int k2 = 0; k2 <= k && first < 0; ++k2) {
        if (!s_ok[k2]) continue;
        bool eq = true;
        for (int l = 0; l < j; ++l) eq &= (drafts[((long long)b * K + k2) * L + l] == code[l]);
        if (eq) first = k2;
      }
    }
    s_new[k] = (ok && first == k) ? 1 : 0;
    __syncthreads();
    if (k == 0) {                                // exclusive scan of the "new node" flags -> slots
      int c = 0;
      for (int i = 0; i < cnt; ++i) { const int f = s_new[i]; s_new[i] = c; c += f; }
      s_cnt = c;
    }
    __syncthreads();
    if (ok) {
      const int slot = s_new[first];
      s_slot[cur][k] = slot;
      if (first == k) {
        const long long s = lvl_bk(e, j, b, slot);
        for (int l = 0; l < L; ++l) e.dw_codes[s * L + l] = l < j ? code[l] : -1;
        e.dw_score[s] = 0.f;
        e.dw_parent[s] = s_slot[prev][k];
      }
    }
    if (k == 0) e.dw_count[(long long)j * e.Bmax + b] = s_cnt;
    __syncthreads();
  }
  if (k == 0) e.d_m[b] = L;
}

// Caller-supplied draft tree (test hook): level j's nodes are taken as listed; a node's parent is the node of level j - 1
// that equals its first j - 1 codes (-1 if there is none: the node is then dead).  One block of >= Kmax threads per request.
__global__ void draft_tree_set_kernel(EngineState e, int batch, int K, const int* tree_codes, const int* tree_count) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x;
  if (b == 0 && threadIdx.x == 0) *e.n_tokens = 0;
  if (b >= batch) return;
  const int L = e.L, k = threadIdx.x;
  const bool row_live = e.row_m[b] < L;
  for (int j = 1; j <= L; ++j) {
    const int cnt = row_live ? max(0, min(tree_count[(long long)(j - 1) * batch + b], K)) : 0;
    const int cnt_prev = j > 1 && row_live ? max(0, min(tree_count[(long long)(j - 2) * batch + b], K)) : 0;
    if (k < cnt) {
      const int* src = tree_codes + (((long long)(j - 1) * batch + b) * K + k) * L;
      const long long s = lvl_bk(e, j, b, k);
      bool ok = true;
      for (int l = 0; l < L; ++l) {
        int c = l < j ? src[l] : -1;
        if (l < j && (c < 0 || c >= e.li.T[l])) { atomicOr(e.status, kStBadCode); ok = false; c = 0; }
        e.dw_codes[s * L + l] = c;
      }
      int parent = j == 1 ? 0 : -1;
      if (ok && j > 1) {
        const int* prv = tree_codes + (((long long)(j - 2) * batch + b) * K) * L;
        for (int k2 = 0; k2 < cnt_prev && parent < 0; ++k2) {
          bool eq = true;
          for (int l = 0; l < j - 1; ++l) eq &= (prv[(long long)k2 * L + l] == src[l]);
          if (eq) parent = k2;
        }
      }
      e.dw_score[s] = 0.f;
      e.dw_parent[s] = ok ? parent : -1;
    }
    if (k == 0) e.dw_count[(long long)j * e.Bmax + b] = cnt;
  }
  if (k == 0) e.d_m[b] = L;
}

// Eq. 2 input: x = h_l + s_l for every (request, beam); s_1 = h_0 (Eq. 1).
template <typename T>
__global__ void draft_x_kernel(EngineState e, int batch, int l, T* x) {
  pdl_wait();
  pdl_launch();
  const int bk = blockIdx.x;                       // b * Kmax + k
  const int b = bk / e.Kmax;
  if (b >= batch) return;
  const float* h = e.h_f32 + ((long long)b * (e.L + 1) + l) * e.d;
  const float* s = (l == 1) ? e.h_f32 + (long long)b * (e.L + 1) * e.d
                            : e.state_lv + ((long long)l * e.Bmax * e.Kmax + bk) * e.d;
  const float uh = e.draft_use_h ? 1.f : 0.f, us = e.draft_use_s ? 1.f : 0.f;     // ablations: drop h_l or s_l
  for (int c = threadIdx.x; c < e.d; c += blockDim.x) x[(long long)bk * e.d + c] = from_f32<T>(uh * h[c] + us * s[c]);
}

// Eq. 3 input rows [s_l ; e_l] for the step s_l -> s_{l+1}.
//   ADD = true (ablation: Transition replaced by addition): writes s_{l+1} = s_l + e_l (fp32) itself, no GEMM follows.
template <typename T, bool ADD>
__global__ void trans_gather_kernel(EngineState e, int batch, int l, const T* embed, T* A) {
  pdl_wait();
  pdl_launch();
  const int bk = blockIdx.x;
  const int b = bk / e.Kmax, k = bk - b * e.Kmax;
  if (b >= batch) return;
  T* dst = A + (long long)bk * 2 * e.d;
  float* nxt = e.state_lv + ((long long)(l + 1) * e.Bmax * e.Kmax + bk) * e.d;
  const auto [parent, code] = draft_source(e, b, k, l);
  const bool live = code >= 0 && parent >= 0;
  if (!live) {
    if (ADD) { for (int c = threadIdx.x; c < e.d; c += blockDim.x) nxt[c] = 0.f; }
    else { for (int c = threadIdx.x; c < 2 * e.d; c += blockDim.x) dst[c] = from_f32<T>(0.f); }
    return;
  }
  const float* s = (l == 1) ? e.h_f32 + (long long)b * (e.L + 1) * e.d
                            : e.state_lv + ((long long)l * e.Bmax * e.Kmax + (long long)b * e.Kmax + parent) * e.d;
  const T* emb = embed + (long long)(e.li.off[l - 1] + code) * e.d;
  for (int c = threadIdx.x; c < e.d; c += blockDim.x) {
    if (ADD) { nxt[c] = s[c] + to_f32(emb[c]); }
    else { dst[c] = from_f32<T>(s[c]); dst[e.d + c] = emb[c]; }
  }
}

// ---- the draft head with merged products ---------------------------------------------------------------------
// s_1 = h_0 (Eq. 1) for every beam slot of every request, as the bf16 A operand of the level's product.
__global__ void draft_state_init_kernel(EngineState e, int batch, __nv_bfloat16* s_act) {
  pdl_wait();
  pdl_launch();
  const int bk = blockIdx.x, b = bk / e.Kmax;
  if (b >= batch) return;
  const float* h0 = e.h_f32 + (long long)b * (e.L + 1) * e.d;
  for (int c = threadIdx.x; c < e.d; c += blockDim.x) s_act[(long long)bk * e.d + c] = __float2bfloat16_rn(h0[c]);
}

// Eq. 3 after the product: s_{l+1}[k] = tanh((W_s s_l)[parent] + (W_e E)[code] + b).  G holds [logits | W_s s_l] of
// every beam slot of level l (W_s s_l from column t_cols on), U = W_e E for every code token.  Which (parent, code) a
// slot takes is decided exactly as in trans_gather_kernel.  per_req: rows of G per request, Kmax (row = the parent's slot), or 1: at
// level 1 every slot's state is s_1 = h_0 (Eq. 1).
__device__ __forceinline__ void draft_state(const EngineState& e, int b, int k, int l, int parent, int code, const float* __restrict__ G,
                                            int per_req, long long g_stride, int t_cols, const float* __restrict__ U,
                                            const float* __restrict__ bias, __nv_bfloat16* s_act, int tid, int n_thr) {
  __nv_bfloat16* dst = s_act + ((long long)b * e.Kmax + k) * e.d;
  if (parent < 0 || code < 0) {                    // no such beam
    for (int c = tid; c < e.d; c += n_thr) dst[c] = __float2bfloat16_rn(0.f);
    return;
  }
  const float* z = G + ((long long)b * per_req + (per_req > 1 ? parent : 0)) * g_stride + t_cols;
  const float* u = U + (long long)(e.li.off[l - 1] + code) * e.d;
#pragma unroll 4
  for (int c = tid; c < e.d; c += n_thr) dst[c] = __float2bfloat16_rn(tanhf(z[c] + u[c] + bias[c]));
}
__device__ __forceinline__ void draft_step_slot(const EngineState& e, int b, int k, int l, const float* __restrict__ G,
                                                int per_req, long long g_stride, int t_cols, const float* __restrict__ U,
                                                const float* __restrict__ bias, __nv_bfloat16* s_act, int tid, int n_thr) {
  const auto [parent, code] = draft_source(e, b, k, l);
  draft_state(e, b, k, l, parent, code, G, per_req, g_stride, t_cols, U, bias, s_act, tid, n_thr);
}
__global__ void draft_step_kernel(EngineState e, int batch, int l, const float* __restrict__ G, int per_req, long long g_stride, int t_cols,
                                  const float* __restrict__ U, const float* __restrict__ bias, __nv_bfloat16* s_act) {
  pdl_wait();
  pdl_launch();
  const int bk = blockIdx.x;
  const int b = bk / e.Kmax, k = bk - b * e.Kmax;
  if (b >= batch) return;
  draft_step_slot(e, b, k, l, G, per_req, g_stride, t_cols, U, bias, s_act, threadIdx.x, blockDim.x);
}
// The selection of draft level l and the state update that follows it, in one launch: a block selects its request's
// beams (or skips that when the request's level is already settled) and then advances the states of its own slots.
template <int VPL>
__global__ void __launch_bounds__(select_max_threads(VPL)) select_step_kernel(SelectArgs a, EngineState e, int l, const float* __restrict__ G,
                                                          int per_req, long long g_stride, int t_cols, const float* __restrict__ U,
                                                          const float* __restrict__ bias, __nv_bfloat16* s_act) {
  pdl_wait();
  pdl_launch();
  const Selected sel = select_body<VPL, false>(a, level_of(a));   // (an earlier level than the last: nothing to probe)
  const int warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5, lane = threadIdx.x & 31;    // a warp per beam slot
  if (sel.active) {                                // (whose selection is still in shared memory: nothing to read back)
    for (int k = warp; k < e.Kmax; k += n_warps)
      draft_state(e, blockIdx.x, k, l, k < sel.n ? sel.r[k] : -1, k < sel.n ? sel.t[k] : -1, G, per_req, g_stride, t_cols, U, bias, s_act, lane, 32);
    return;
  }
  for (int k = warp; k < e.Kmax; k += n_warps)
    draft_step_slot(e, blockIdx.x, k, l, G, per_req, g_stride, t_cols, U, bias, s_act, lane, 32);
}

// dst[b, r, :] = src[(b * row_mul + r), 0 : T] + bias[b, :]
__global__ void copy_logits_bias_kernel(const float* src, long long row_stride, int row_mul, int n_beams, int T,
                                        const float* bias, long long bias_stride, float* dst) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x / n_beams, r = blockIdx.x % n_beams;
  const float* z = src + ((long long)b * row_mul + r) * row_stride;
  for (int t = threadIdx.x; t < T; t += blockDim.x) dst[(long long)blockIdx.x * T + t] = z[t] + bias[(long long)b * bias_stride + t];
}

// Eq. 4 on the first n codes: two tuples of valid codes agree on them exactly when these keys are equal.
__device__ __forceinline__ unsigned long long prefix_key_of(const EngineState& e, const int* codes, int n) {
  unsigned long long k = 0;
  for (int l = 0; l < n; ++l) k += (unsigned long long)(unsigned)codes[l] * e.li.mult[l];
  return k;
}

// ----------------------------------------------------------------------------------------------------
// verify-pass token list (the nodes M_p runs on this round)
// ----------------------------------------------------------------------------------------------------
// Request with m levels settled: nodes = the level-m code of every beam of B_m (slot = beam rank) and, for the levels
// m+1..L-1, the last code of every alive node of the round's draft tree (slot = the node's slot in its level): one token
// per distinct drafted prefix.  A level-m node of the tree is alive if its codes are a beam of B_m; a higher node if its
// parent is alive.  Tokens of a request are contiguous; the requests take their place in the list in the order in which
// their blocks get there (no row of a pass depends on where it stands).
__device__ __forceinline__ void nodes_body(const EngineState& e) {
  const int b = blockIdx.x;
  const int L = e.L, Kmax = e.Kmax;
  __shared__ int s_off, n_alive, s_rank[kMaxLevels][128], s_level_start[kMaxLevels + 1];
  __shared__ unsigned long long s_key[128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  const int m = e.row_m[b];
  if (b == 0 && threadIdx.x == 0) *e.draft_rows = 0;     // this round's drafting is over; round_end raises it again if needed
  if (m >= L) {
    if (threadIdx.x == 0) { e.row_tok_count[b] = 0; e.row_cur[b] = -1; e.req_info[b] = make_int4(0, 0, b, 0); }
    return;
  }
  const int nb = e.tb_count[m * e.Bmax + b];
  if (threadIdx.x == 0) n_alive = 0;
  for (int r = threadIdx.x; r < nb; r += blockDim.x) s_key[r] = prefix_key_of(e, e.tb_codes + lvl_bk(e, m, b, r) * L, m);
  __syncthreads();
  for (int j = m; j < L; ++j) {
    const int cnt = min(e.dw_count[(long long)j * e.Bmax + b], Kmax);
    for (int k = threadIdx.x; k < Kmax; k += blockDim.x) {
      int beta = -1;
      if (k < cnt) {
        if (j == m) {
          const unsigned long long key = prefix_key_of(e, e.dw_codes + lvl_bk(e, m, b, k) * L, m);
          for (int r = nb - 1; r >= 0; --r)
            if (s_key[r] == key) beta = r;
        } else {
          const int p = e.dw_parent[lvl_bk(e, j, b, k)];
          if (p >= 0 && p < Kmax) beta = e.d_beam[lvl_bk(e, j - 1, b, p)];
          if (beta >= 0) atomicAdd(&n_alive, 1);
        }
      }
      e.d_beam[lvl_bk(e, j, b, k)] = beta;
    }
    __syncthreads();                               // level j's answers (global, this block's own) before level j + 1 reads them
  }
  if (threadIdx.x == 0) {
    const int n_tok = nb + n_alive, off = atomicAdd(e.n_tokens, n_tok);
    s_off = off;
    e.row_tok_count[b] = n_tok; e.row_tok_start[b] = off;
    e.row_cur[b] = m; e.row_m_start[b] = m;
    e.req_info[b] = make_int4(off, n_tok, b, n_tok > 0 ? e.row_P[b] : 0);
  }
  for (int i = threadIdx.x; i < L * Kmax; i += blockDim.x) e.node_index[(long long)b * L * Kmax + i] = -1;
  // rank of every alive node within its level (a warp per level: ballots over its <= 128 slots)
  for (int j = m + 1 + warp; j < L; j += n_warps) {
    int base = 0;
    for (int k0 = 0; k0 < Kmax; k0 += 32) {
      const int k = k0 + lane;
      const bool alive = k < Kmax && k < e.dw_count[(long long)j * e.Bmax + b] && e.d_beam[lvl_bk(e, j, b, k)] >= 0;
      const unsigned mask = __ballot_sync(0xffffffffu, alive);
      if (k < 128) s_rank[j][k] = alive ? base + __popc(mask & ((1u << lane) - 1u)) : -1;
      base += __popc(mask);
    }
    if (lane == 0) s_level_start[j] = base;        // the level's count for now; turned into a start below
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int start = nb;
    for (int j = m + 1; j < L; ++j) { const int c = s_level_start[j]; s_level_start[j] = start; start += c; }
  }
  __syncthreads();
  const int P = e.row_P[b];
  const long long slab_elems = (long long)Kmax * e.Hkv * e.hd;       // one level slab of one request
  const long long row_elems = (long long)(L - 1) * slab_elems;
  auto kv_off = [&](int level, int slot) {                             // level 1..L-1
    return (long long)b * row_elems + (long long)(level - 1) * slab_elems + (long long)slot * e.Hkv * e.hd;
  };
  // level-m nodes: the true beams
  for (int r = threadIdx.x; r < nb; r += blockDim.x) {
    const int t = s_off + r;
    const long long bi = lvl_bk(e, m, b, r);
    e.tok_row[t] = b; e.tok_pos[t] = P + m - 1; e.tok_ctx_len[t] = P;
    e.tok_id[t] = e.li.off[m - 1] + e.tb_codes[bi * L + (m - 1)];
    e.tok_kv_dst[t] = kv_off(m, r);
    for (int i = 1; i <= L; ++i) {
      long long o = -1;
      if (i < m) o = kv_off(i, e.tb_anc[bi * L + (i - 1)]);
      else if (i == m) o = kv_off(m, r);
      e.tok_ext[(long long)t * L + (i - 1)] = o;
    }
    e.tb_src[bi] = t;
    e.tb_self[bi] = r;
    e.node_index[((long long)b * L + m) * Kmax + r] = t;
  }
  // levels m+1 .. L-1: the alive nodes of the draft tree
  const int n_lv = L - 1 - m;
  for (int idx = threadIdx.x; idx < n_lv * Kmax; idx += blockDim.x) {
    const int j = m + 1 + idx / Kmax, k = idx % Kmax;
    const int rank = s_rank[j][k];
    if (rank < 0) continue;
    const int t = s_off + s_level_start[j] + rank;
    const int beta = e.d_beam[lvl_bk(e, j, b, k)];
    const long long bi = lvl_bk(e, m, b, beta);
    const long long di = lvl_bk(e, j, b, k);
    e.tok_row[t] = b; e.tok_pos[t] = P + j - 1; e.tok_ctx_len[t] = P;
    e.tok_id[t] = e.li.off[j - 1] + e.dw_codes[di * L + (j - 1)];
    e.tok_kv_dst[t] = kv_off(j, k);
    int anc[kMaxLevels + 1];                       // anc[i] = slot of the node's ancestor of level i in the tree
    anc[j] = k;
    for (int i = j; i > m + 1; --i) anc[i - 1] = e.dw_parent[lvl_bk(e, i, b, anc[i])];
    for (int i = 1; i <= L; ++i) {
      long long o = -1;
      if (i < m) o = kv_off(i, e.tb_anc[bi * L + (i - 1)]);
      else if (i == m) o = kv_off(m, beta);
      else if (i <= j) o = kv_off(i, anc[i]);
      e.tok_ext[(long long)t * L + (i - 1)] = o;
    }
    e.node_index[((long long)b * L + j) * Kmax + k] = t;
  }
}

__global__ void __launch_bounds__(128) nodes_kernel(EngineState e) {
  pdl_wait();
  pdl_launch();
  nodes_body(e);
}
// The draft head's last selection, whose tuples nothing asks for before the round's end, and beside it (blockIdx.y = 1) the token
// list, which goes by the levels before.
template <int VPL, bool PROBE>
__global__ void __launch_bounds__(select_max_threads(VPL)) select_nodes_kernel(SelectArgs a, EngineState e) {
  pdl_wait();
  pdl_launch();
  if (blockIdx.y == 0) select_body<VPL, PROBE>(a, level_of(a));
  else nodes_body(e);
}

// Teacher-forced nodes: beams given by the caller, every beam processes all of its `level` codes.
__global__ void nodes_from_prefixes_kernel(EngineState e, int batch, int n_beams, int level, const int* prefixes) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x;
  const int L = e.L, Kmax = e.Kmax;
  const int per_row = n_beams * level;
  const int P = e.row_P[b];
  const long long slab_elems = (long long)Kmax * e.Hkv * e.hd;
  const long long row_elems = (long long)(L - 1) * slab_elems;
  if (b == 0 && threadIdx.x == 0) *e.n_tokens = batch * per_row;
  if (threadIdx.x == 0) {
    e.row_tok_start[b] = b * per_row; e.row_tok_count[b] = per_row;
    e.req_info[b] = make_int4(b * per_row, per_row, b, P);
  }
  for (int i = threadIdx.x; i < L * Kmax; i += blockDim.x) e.node_index[(long long)b * L * Kmax + i] = -1;
  __syncthreads();
  for (int idx = threadIdx.x; idx < per_row; idx += blockDim.x) {
    const int j = 1 + idx / n_beams, r = idx % n_beams;
    const int t = b * per_row + idx;
    int code = prefixes[((long long)b * n_beams + r) * level + (j - 1)];
    if (code < 0 || code >= e.li.T[j - 1]) { atomicOr(e.status, kStBadCode); code = 0; }
    e.tok_row[t] = b; e.tok_pos[t] = P + j - 1; e.tok_ctx_len[t] = P;
    e.tok_id[t] = e.li.off[j - 1] + code;
    const long long self = (long long)b * row_elems + (long long)(j - 1) * slab_elems + (long long)r * e.Hkv * e.hd;
    e.tok_kv_dst[t] = self;
    for (int i = 1; i <= L; ++i)
      e.tok_ext[(long long)t * L + (i - 1)] =
          (i <= j) ? (long long)b * row_elems + (long long)(i - 1) * slab_elems + (long long)r * e.Hkv * e.hd : -1;
    e.node_index[((long long)b * L + j) * Kmax + r] = t;
  }
}

// ----------------------------------------------------------------------------------------------------
// accept / roll back (Algorithm 2's rejection and update steps)
// ----------------------------------------------------------------------------------------------------
// The fused kernel reads all it may need about its request at its start, under the selection, into shared memory: each
// dependent read behind the selection would be an L2 round trip of 0.6 us in a kernel of 13 (and there were up to 14).
struct AdvanceSmem {
  unsigned long long* key;       // [L][Kmax] keys of the alive nodes of level n + 1 (row 0), then of the beams of levels 1..L
  int* codes;                    // [Kmax][L] tb_codes of level n
  int* node;                     // [Kmax][L] dw_codes of level n + 1
  int *dbeam, *nidx, *self;      // [Kmax]    d_beam and node_index of level n + 1, tb_self of level n
  int* anc;                      // [Kmax][L] tb_anc of level n
  int* drafted;                  // [Kmax][L] dw_codes of level L (the round's end only, like what follows)
  int* beams;                    // [L][Kmax][L] tb_codes of levels 1..L
};
__device__ __forceinline__ AdvanceSmem advance_smem(unsigned char* base, int Kmax, int L) {
  AdvanceSmem m;
  m.key = reinterpret_cast<unsigned long long*>(base);
  m.codes = reinterpret_cast<int*>(m.key + (size_t)L * Kmax);
  m.node = m.codes + Kmax * L; m.anc = m.node + Kmax * L;
  m.dbeam = m.anc + Kmax * L; m.nidx = m.dbeam + Kmax; m.self = m.nidx + Kmax;
  m.drafted = m.self + Kmax; m.beams = m.drafted + Kmax * L;
  return m;
}

// After B_{n+1} has been selected for a request whose beams B_n had logits in this pass (sel.active):
//   n + 1 == L : the request is finished; B_L is the result.
//   otherwise  : every beam of B_{n+1} inherits its parent's KV slots (a slot-table rewrite: rejected drafts'
//                KV rows simply become unreachable) and is matched against the alive nodes of level n+1 of the draft
//                tree.  If every beam is such a node, its hidden state is already in the pass and selection goes on;
//                else level n+1 is the rejection level and the request waits for the next round.
// nd: nodes of level n + 1.  Returns where the request stands: levels settled, and the level whose beams have logits in this pass (or -1).
struct Advanced { int m, cur; };
__device__ __forceinline__ Advanced advance_body(const EngineState& e, const AdvanceSmem& sm, const Selected& sel, int n, int K, int nd,
                                             int* out_codes, float* out_score, int* out_count) {
  const int b = blockIdx.x, L = e.L, n1 = n + 1, cnt = sel.n;
  if (n1 == L) {
    for (int k = threadIdx.x; k < K; k += blockDim.x) out_score[(long long)b * K + k] = k < cnt ? sel.s[k] : -INFINITY;
    for (int i = threadIdx.x; i < K * L; i += blockDim.x) {
      const int k = i / L, l = i - k * L;
      out_codes[(long long)b * K * L + i] = k >= cnt ? -1 : l < n ? sm.codes[sel.r[k] * L + l] : sel.t[k];
    }
    if (threadIdx.x == 0) { out_count[b] = cnt; e.row_m[b] = L; e.row_cur[b] = -1; }
    return Advanced{L, -1};
  }
  __shared__ int all_matched;
  if (threadIdx.x == 0) all_matched = 1;
  for (int k = threadIdx.x; k < nd; k += blockDim.x)           // (a dead node: no key)
    sm.key[k] = sm.dbeam[k] < 0 ? kEmptyKey : prefix_key_of(e, sm.node + k * L, n1);
  __syncthreads();
  for (int r = threadIdx.x; r < cnt; r += blockDim.x) {
    const long long bi = lvl_bk(e, n1, b, r);
    const int parent = sel.r[r];
    for (int i = 0; i + 1 < n; ++i) e.tb_anc[bi * L + i] = sm.anc[parent * L + i];
    if (n >= 1) e.tb_anc[bi * L + (n - 1)] = sm.self[parent];
    const unsigned long long key = prefix_key_of(e, sm.codes + parent * L, n) + (unsigned long long)sel.t[r] * e.li.mult[n];
    int match = -1;
    for (int k = nd - 1; k >= 0; --k)
      if (sm.key[k] == key) match = k;
    e.tb_src[bi] = match >= 0 ? sm.nidx[match] : -1;
    e.tb_self[bi] = match;
    if (match < 0) all_matched = 0;
  }
  __syncthreads();
  const Advanced ad{cnt == 0 ? L : n1, (all_matched && cnt > 0) ? n1 : -1};   // (no beam survived -- possible only with an empty codebook:
  if (threadIdx.x == 0) {                                                       //  finish empty)
    e.row_m[b] = ad.m;
    e.row_cur[b] = ad.cur;
    if (cnt == 0) out_count[b] = 0;
  }
  return ad;
}

// End of a round: accepted length of every draft = the largest i <= (level reached) with D[k][0..i) in B_i;
// trace outputs; the request's own counters (unfinished, primary tokens, accepted levels, drafted tuples) and, once, the status word
// straight to the host's pinned memory: no block waits for another or for the bus.  (Added up on the device, with the last block copying
// the sums from one thread behind a system-wide fence, this took 11 us of a round.)
// adaptive: a request whose round settled only the one level that the pass settles anyway gained nothing from its drafts
// and stops drafting (its remaining rounds are plain autoregressive steps).
// re.draft_next: the start of the next round's drafting (Algorithm 2's drafting step): the draft head continues from the true beams B_m.
// What the block read about its request at the start of the kernel:
struct RowState { int m, m_start, spec, tokens, nd_last; };    // nd_last: drafted tuples (nodes of level L)
__device__ __forceinline__ void round_end_body(const EngineState& e, const AdvanceSmem& sm, int m_now, const RowState& rs, int K,
                                               const RoundEnd& re) {
  const int b = blockIdx.x, batch = gridDim.x, round = re.round;
  const int L = e.L, Kmax = e.Kmax;
  const nezha_trace& tr = re.tr;
  __shared__ int acc_sum;
  const int took_part = rs.tokens > 0;
  const int nd = took_part ? rs.nd_last : 0;
  const long long tro = ((long long)(round - 1) * batch + b);
  if (threadIdx.x == 0) acc_sum = 0;
  // thread k answers for drafted tuple k (K <= 128 <= threads)
  const int k = threadIdx.x;
  const bool mine = k < K && k < nd;
  int acc = mine ? 0 : -1;
  if (nd > 0) {
    for (int i = threadIdx.x; i < m_now * Kmax; i += blockDim.x) {
      const int lv = i / Kmax, r = i - lv * Kmax;  // beams of level lv + 1 (beyond their count -- at most K -- the codes are -1)
      sm.key[i] = r < K && sm.beams[(lv * Kmax + r) * L] >= 0 ? prefix_key_of(e, sm.beams + (lv * Kmax + r) * L, lv + 1) : kEmptyKey;
    }
    __syncthreads();
    unsigned long long key = 0;
    for (int i = 1; i <= m_now && mine && acc == i - 1; ++i) {
      key += (unsigned long long)(unsigned)sm.drafted[k * L + i - 1] * e.li.mult[i - 1];
      bool in = false;
      for (int r = 0; r < K; ++r) in |= sm.key[(i - 1) * Kmax + r] == key;
      if (in) acc = i;
    }
  }
  __syncthreads();
  if (mine && acc > 0) atomicAdd(&acc_sum, acc);
  if (k < K) {
    if (tr.accepted_len) tr.accepted_len[tro * K + k] = acc;
    if (tr.drafts)
      for (int l = 0; l < L; ++l)
        tr.drafts[(tro * K + k) * L + l] = (k < nd) ? sm.drafted[k * L + l] : -1;
    if (tr.tree_codes)
      for (int j = 1; j <= L; ++j) {
        const int nj = took_part ? min(e.dw_count[(long long)j * e.Bmax + b], Kmax) : 0;
        const long long o = ((((long long)(round - 1) * L + (j - 1)) * batch + b) * K + k) * L;
        for (int l = 0; l < L; ++l) tr.tree_codes[o + l] = (k < nj && l < j) ? e.dw_codes[lvl_bk(e, j, b, k) * L + l] : -1;
      }
  }
  if (tr.tree_count && threadIdx.x < L)
    tr.tree_count[((long long)(round - 1) * L + threadIdx.x) * batch + b] =
        took_part ? min(min(e.dw_count[(long long)(threadIdx.x + 1) * e.Bmax + b], Kmax), K) : -1;
  __syncthreads();                                 // (the round's draft tree has been read)
  const int spec = took_part && re.adaptive ? (m_now - rs.m_start >= 2 ? 1 : 0) : rs.spec;
  if (re.draft_next) {
    const bool drafts = m_now < L && spec;         // (not finished, and its drafting not switched off; otherwise an empty tree)
    if (drafts) {
      const int cnt = e.tb_count[(long long)m_now * e.Bmax + b];
      for (int i = threadIdx.x; i < Kmax * (L + 1); i += blockDim.x) {
        const int s = i / (L + 1), l = i - s * (L + 1);
        const long long o = lvl_bk(e, m_now, b, s);
        const bool live = s < cnt;
        if (l < L) e.dw_codes[o * L + l] = live ? sm.beams[((m_now - 1) * Kmax + s) * L + l] : -1;
        else { e.dw_score[o] = live ? e.tb_score[o] : -INFINITY; e.dw_parent[o] = live ? s : -1; }
      }
      if (threadIdx.x == 0) { e.dw_count[(long long)m_now * e.Bmax + b] = cnt; e.d_m[b] = m_now; }
    } else {
      if (threadIdx.x == 0) e.d_m[b] = L;
      if ((int)threadIdx.x <= L) e.dw_count[(long long)threadIdx.x * e.Bmax + b] = 0;
    }
  }
  if (threadIdx.x == 0) {
    if (tr.n_draft) tr.n_draft[tro] = took_part ? nd : -1;
    if (tr.level_reached) tr.level_reached[tro] = took_part ? m_now : -1;
    if (took_part && re.adaptive) e.row_spec[b] = spec;
    if (m_now < L && spec) atomicMax(e.draft_rows, batch * Kmax);            // somebody drafts next round
    if (b == 0) *e.n_tokens = 0;                   // for the next round's token list
    re.rows[b] = make_int4(m_now < L ? 1 : 0, took_part ? rs.tokens : 0, acc_sum, nd);
  }
  if (b == 0 && threadIdx.x < 4) re.host[threadIdx.x] = *(volatile int*)(e.status + threadIdx.x);
}

// A pass's selections of a request, one level after the other for as long as its beams are nodes of the pass: B_{n+1} from the logits
// of B_n, the step above, and on with n + 1 -- and, behind the last, the end of the round.  One launch: with a launch per level the
// levels that a rejection leaves over were launches for nothing (64 requests, small shape, natural drafts: three of seven).
// a: the arguments of the first level; levels: the levels from there on up to (not including) `last`.
template <int VPL, bool PROBE>
__global__ void __launch_bounds__(select_max_threads(VPL)) select_advance_kernel(SelectArgs a, EngineState e, int last, int K, int* out_codes,
                                                             float* out_score, int* out_count, RoundEnd re, int select_bytes) {
  extern __shared__ unsigned char smem_raw[];
  const int b = blockIdx.x, L = e.L, Kmax = e.Kmax;
  const AdvanceSmem sm = advance_smem(smem_raw + select_bytes, Kmax, L);
  pdl_wait();
  pdl_launch();
  auto fetch_beams = [&](int lv) { cp_async_ints(sm.beams + (lv - 1) * Kmax * L, e.tb_codes + lvl_bk(e, lv, b, 0) * L, Kmax * L); };
  RowState rs{0, 0, 0, 0, 0};
  if (re.host) {
    cp_async_ints(sm.drafted, e.dw_codes + lvl_bk(e, L, b, 0) * L, Kmax * L);
    for (int lv = 1; lv <= L; ++lv) fetch_beams(lv);
    rs = RowState{e.row_m[b], e.row_m_start[b], e.row_spec[b], e.row_tok_count[b], min(e.dw_count[(long long)L * e.Bmax + b], Kmax)};
  }
  int m_now = rs.m;
  SelectLevel v = level_of(a);
#pragma unroll 1
  for (;;) {
    const int n = v.n, n1 = n + 1;
    cp_async_ints(sm.codes, e.tb_codes + lvl_bk(e, n, b, 0) * L, Kmax * L);
    cp_async_ints(sm.node, e.dw_codes + lvl_bk(e, n1, b, 0) * L, Kmax * L);
    if (n1 < L) {
      cp_async_ints(sm.dbeam, e.d_beam + lvl_bk(e, n1, b, 0), Kmax);
      cp_async_ints(sm.nidx, e.node_index + ((long long)b * L + n1) * Kmax, Kmax);
      cp_async_ints(sm.self, e.tb_self + lvl_bk(e, n, b, 0), Kmax);
      cp_async_ints(sm.anc, e.tb_anc + lvl_bk(e, n, b, 0) * L, Kmax * L);
    }
    const int nd = min(e.dw_count[(long long)n1 * e.Bmax + b], Kmax);
    const Selected sel = select_body<VPL, PROBE>(a, v, sm.codes);
    int cur = sel.gate;                            // where an inactive request stands: not here, or further on
    if (sel.active) {
      const Advanced ad = advance_body(e, sm, sel, n, K, nd, out_codes, out_score, out_count);
      m_now = ad.m; cur = ad.cur;
    } else {
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncthreads();                               // the tables that this level has written and the next reads, and shared memory
    if (re.host && sel.active) fetch_beams(n1);    // (as they are now)
    if (cur < n1 || n1 >= last) break;
    // on to level n1
    const long long lv = (long long)e.Bmax * Kmax;
    v.col_off += v.T;
    v.n = n1; v.T = e.li.T[n1]; v.per_beam = v.T; v.gate_value = n1;
    v.filter = n1 + 1 == L ? 1 : 0;
    if (v.filter) v.prefix_filter = 0;
    v.src_row += lv; v.in_codes += lv * L; v.in_score += lv; v.in_count += e.Bmax;
    v.out_codes += lv * L; v.out_score += lv; v.out_parent += lv; v.out_count += e.Bmax;
  }
  if (re.host) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    round_end_body(e, sm, m_now, rs, K, re);
  }
}

// dst[b, r, :] = src[row(b, r), col_off : col_off + T],
// row = row_index ? row_index[b*idx_stride + r] : b*row_mul + r*beam_mul
__global__ void copy_logits_kernel(const float* src, long long row_stride, int col_off, const int* row_index, int row_mul,
                                   int beam_mul, int n_beams, int idx_stride, int T, float* dst) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x / n_beams, r = blockIdx.x % n_beams;
  const long long row = row_index ? row_index[(long long)b * idx_stride + r] : (long long)b * row_mul + (long long)r * beam_mul;
  if (row < 0) return;
  for (int t = threadIdx.x; t < T; t += blockDim.x)
    dst[(long long)blockIdx.x * T + t] = src[row * row_stride + col_off + t];
}

__global__ void trace_beams_kernel(EngineState e, int batch, int K, nezha_trace tr) {
  pdl_wait();
  pdl_launch();
  const int b = blockIdx.x;
  const int L = e.L;
  for (int n = 1; n <= L; ++n) {
    const int cnt = e.tb_count[n * e.Bmax + b];
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
      const long long s = lvl_bk(e, n, b, k);
      const long long o = ((long long)(n - 1) * batch + b) * K + k;
      if (tr.beam_scores) tr.beam_scores[o] = k < cnt ? e.tb_score[s] : -INFINITY;
      if (tr.beams)
        for (int l = 0; l < L; ++l) tr.beams[o * L + l] = (k < cnt && l < n) ? e.tb_codes[s * L + l] : -1;
    }
  }
}

}  // namespace

void launch_fill_i32(int* p, long long n, int v, cudaStream_t st) {
  if (n <= 0) return;
  LaunchScope ls(kcMisc, st);
  launch_pdl(fill_i32_kernel, dim3((unsigned)((n + 255) / 256 < 1184 ? (n + 255) / 256 : 1184)), dim3(256), 0, st, p, n, v);
}
void launch_decode_begin(const EngineState& e, int batch, int K, int from_scratch, int* out_codes, float* out_scores, int* out_count,
                         const nezha_trace& tr, cudaStream_t st) {
  LaunchScope ls(kcMisc, st);
  launch_pdl(decode_begin_kernel, dim3(batch), dim3(128), 0, st, e, batch, K, from_scratch, out_codes, out_scores, out_count, tr);
}
void launch_draft_set(const EngineState& e, int batch, int K, const int* drafts, const int* n_draft, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  launch_pdl(draft_set_kernel, dim3(batch), dim3(128), 0, st, e, batch, K, drafts, n_draft);
}
void launch_draft_tree_set(const EngineState& e, int batch, int K, const int* tree_codes, const int* tree_count, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  launch_pdl(draft_tree_set_kernel, dim3(batch), dim3(128), 0, st, e, batch, K, tree_codes, tree_count);
}
void launch_draft_x(const EngineState& e, int batch, int l, void* x, bool bf16, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  if (bf16) launch_pdl(draft_x_kernel<__nv_bfloat16>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, (__nv_bfloat16*)x);
  else launch_pdl(draft_x_kernel<float>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, (float*)x);
}
void launch_trans_gather(const EngineState& e, int batch, int l, const void* embed, void* A, bool bf16,
                         cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  if (bf16)
    launch_pdl(trans_gather_kernel<__nv_bfloat16, false>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, (const __nv_bfloat16*)embed,
                                                                      (__nv_bfloat16*)A);
  else launch_pdl(trans_gather_kernel<float, false>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, (const float*)embed, (float*)A);
}
void launch_trans_add(const EngineState& e, int batch, int l, const void* embed, bool bf16, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  if (bf16)
    launch_pdl(trans_gather_kernel<__nv_bfloat16, true>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l,
               (const __nv_bfloat16*)embed, (__nv_bfloat16*)nullptr);
  else
    launch_pdl(trans_gather_kernel<float, true>, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, (const float*)embed,
               (float*)nullptr);
}
void launch_draft_state_init(const EngineState& e, int batch, void* s_act, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  launch_pdl(draft_state_init_kernel, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, (__nv_bfloat16*)s_act);
}
void launch_draft_step(const EngineState& e, int batch, int l, const float* G, int per_req, long long g_stride, int t_cols, const float* U,
                       const float* bias, void* s_act, cudaStream_t st) {
  LaunchScope ls(kcDraftGlue, st);
  launch_pdl(draft_step_kernel, dim3(batch * e.Kmax), dim3(128), 0, st, e, batch, l, G, per_req, g_stride, t_cols, U, bias,
             (__nv_bfloat16*)s_act);
}
size_t advance_smem_bytes(int Kmax, int L) { return (size_t)Kmax * (8 * L + 4 * (4 * L + 3 + L * L)); }
cudaError_t select_step_configure(int bytes) {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto vpl) {
    constexpr int V = decltype(vpl)::value;
    constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_advance_kernel<V, false>, attr, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_advance_kernel<V, true>, attr, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_step_kernel<V>, attr, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_nodes_kernel<V, false>, attr, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(select_nodes_kernel<V, true>, attr, bytes);
  };
  set(Vpl<1>{}); set(Vpl<8>{}); set(Vpl<16>{}); set(Vpl<32>{});
  return e;
}
void launch_select_step(const SelectArgs& a, const EngineState& e, int l, const float* G, int per_req, long long g_stride, int t_cols,
                        const float* U, const float* bias, void* s_act, cudaStream_t st) {
  if (a.batch <= 0) return;
  const size_t smem = select_smem_bytes(a.in_stride, a.K);
  LaunchScope ls(kcSelect, st);
  const int warps = select_warps(a);
  const dim3 block(32 * warps), grid(a.batch);
  __nv_bfloat16* s = (__nv_bfloat16*)s_act;
  with_vpl(a.T, [&](auto vpl) {
    launch_pdl(select_step_kernel<decltype(vpl)::value>, grid, block, smem, st, a, e, l, G, per_req, g_stride, t_cols, U, bias, s);
  });
}
void launch_copy_logits_bias(const float* src, long long row_stride, int row_mul, int batch, int n_beams, int T,
                             const float* bias, long long bias_stride, float* dst, cudaStream_t st) {
  LaunchScope ls(kcMisc, st);
  launch_pdl(copy_logits_bias_kernel, dim3(batch * n_beams), dim3(128), 0, st, src, row_stride, row_mul, n_beams, T, bias,
             bias_stride, dst);
}
void launch_build_nodes(const EngineState& e, int batch, cudaStream_t st) {
  LaunchScope ls(kcNodes, st);
  launch_pdl(nodes_kernel, dim3(batch), dim3(128), 0, st, e);
}
void launch_select_nodes(const SelectArgs& a, const EngineState& e, cudaStream_t st) {
  if (a.batch <= 0) return;
  const size_t smem = select_smem_bytes(a.in_stride, a.K);
  LaunchScope ls(kcSelect, st);
  const dim3 block(32 * select_warps(a)), grid(a.batch, 2);
  with_vpl(a.T, [&](auto vpl) {
    constexpr int V = decltype(vpl)::value;
    launch_pdl(select_probes(a) ? select_nodes_kernel<V, true> : select_nodes_kernel<V, false>, grid, block, smem, st, a, e);
  });
}
void launch_nodes_from_prefixes(const EngineState& e, int batch, int n_beams, int level, const int* prefixes,
                                cudaStream_t st) {
  LaunchScope ls(kcNodes, st);
  launch_pdl(nodes_from_prefixes_kernel, dim3(batch), dim3(128), 0, st, e, batch, n_beams, level, prefixes);
}
void launch_select_advance(const SelectArgs& a, const EngineState& e, int last, int K, int* out_codes, float* out_score,
                           int* out_count, const RoundEnd& re, cudaStream_t st) {
  if (a.batch <= 0) return;
  const size_t select_bytes = select_smem_bytes(a.in_stride, a.K), smem = select_bytes + advance_smem_bytes(e.Kmax, e.L);
  LaunchScope ls(kcSelect, st);
  SelectArgs widest = a;                           // (of the levels: the codes per lane and the warps)
  for (int n = a.n + 1; n < last; ++n) widest.T = a.li.T[n] > widest.T ? a.li.T[n] : widest.T;
  SelectArgs final_level = a;
  final_level.filter = last == e.L ? 1 : 0; final_level.per_beam = final_level.T;
  if (final_level.filter) final_level.prefix_filter = 0;
  const dim3 block(32 * select_warps(widest)), grid(a.batch);
  with_vpl(widest.T, [&](auto vpl) {
    constexpr int V = decltype(vpl)::value;
    launch_pdl(select_probes(final_level) ? select_advance_kernel<V, true> : select_advance_kernel<V, false>, grid, block, smem, st, a, e,
               last, K, out_codes, out_score, out_count, re, (int)select_bytes);
  });
}
void launch_copy_logits(const float* src, long long row_stride, int col_off, const int* row_index, int row_mul,
                        int beam_mul, int batch, int n_beams, int idx_stride, int T, float* dst, cudaStream_t st) {
  LaunchScope ls(kcMisc, st);
  launch_pdl(copy_logits_kernel, dim3(batch * n_beams), dim3(128), 0, st, src, row_stride, col_off, row_index, row_mul, beam_mul, n_beams,
                                                      idx_stride, T, dst);
}

// Prompt tokens of a chunk of requests: [BOS, history codes item by item, SP_1..SP_L], request after request with nothing in
// between.  A call whose histories are of unequal length is given rows of max_n items, but a pass over all of them would
// spend on padding what the longest history costs for every request; the token list holds the real tokens only and its
// length stays on the device (pf_n_tokens: the row count of every kernel of the pass).  Grid = (requests, tiles of 256
// positions); a block adds up the lengths of the requests before its own (a few thousand at most, one round of loads).
__global__ void __launch_bounds__(256) prefill_tokens_kernel(EngineState e, const int* hist, const int* n_hist, int b0, int rows,
                                                             int max_n, int S_cap, int* h_rows) {
  pdl_wait();
  pdl_launch();
  const int lb = blockIdx.x, b = b0 + lb, L = e.L;
  auto items = [&](int row) {
    const int nh = n_hist[b0 + row];
    return nh < 0 ? 0 : nh > max_n ? max_n : nh;
  };
  __shared__ int part[8];
  int before = 0;
  for (int i = threadIdx.x; i < lb; i += blockDim.x) before += items(i);
  before = (int)__reduce_add_sync(0xffffffffu, (unsigned)before);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = before;
  __syncthreads();
  before = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) before += part[i];
  const int nh = items(lb), P = 1 + nh * L, S = P + L;
  const int start = lb * (1 + L) + before * L;     // first token of the request in the list
  const int p = blockIdx.y * blockDim.x + threadIdx.x;
  if (p == 0) {
    if (n_hist[b] != nh) atomicOr(e.status, kStBadCode);
    e.row_P[b] = P; e.pf_row_start[lb] = start; e.pf_row_count[lb] = S;
    e.pf_req_info[lb] = make_int4(start, S, b, -1);
    if (lb == rows - 1) *e.pf_n_tokens = start + S;
  }
  if (p >= S) return;
  const int idx = start + p;
  int tok = e.li.vocab_codes + L;                  // BOS
  if (p >= P) {
    tok = e.li.vocab_codes + (p - P);
  } else if (p > 0) {
    const int item = (p - 1) / L, lv = (p - 1) % L;
    int code = hist[((long long)b * max_n + item) * L + lv];
    if (code < 0 || code >= e.li.T[lv]) { atomicOr(e.status, kStBadCode); code = 0; }
    tok = e.li.off[lv] + code;
  }
  e.tok_id[idx] = tok; e.tok_pos[idx] = p; e.tok_row[idx] = b; e.tok_ctx_len[idx] = p + 1;
  e.tok_kv_dst[idx] = ((long long)b * e.Hkv * S_cap + p) * e.hd;
  if (p >= P - 1) h_rows[lb * (L + 1) + (p - (P - 1))] = idx;
}

void launch_prefill_tokens(const EngineState& e, const int* hist, const int* n_hist, int b0, int rows, int max_n,
                           int S_call, int S_cap, int* h_rows, cudaStream_t st) {
  LaunchScope ls(kcNodes, st);
  launch_pdl(prefill_tokens_kernel, dim3(rows, (S_call + 255) / 256), dim3(256), 0, st, e, hist, n_hist, b0, rows, max_n, S_cap, h_rows);
}
void launch_trace_beams(const EngineState& e, int batch, int K, const nezha_trace& tr, cudaStream_t st) {
  LaunchScope ls(kcMisc, st);
  launch_pdl(trace_beams_kernel, dim3(batch), dim3(64), 0, st, e, batch, K, tr);
}

}  // namespace nz
