// Shared declarations of the decode library's translation units (device helpers, argument structs,
// kernel launchers).  Everything here is internal; the public surface is include/nezha.h.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "nezha.h"

namespace nz {

constexpr int kMaxLevels = NEZHA_MAX_LEVELS;
constexpr int kBucketBytes = 32;                 // one sector per bucket of the hash set: 4 wide or 8 narrow slots
constexpr unsigned long long kEmptyKey = ~0ull;  // never a packed key: prod(T) < 2^64 - 1
constexpr int kMaxProbeBuckets = 4096;           // bound of every probe / insert walk

// bits of the device status word
enum : int { kStHashFull = 1, kStBadCode = 2, kStInternal = 4 };

// Kernel classes for the launch counter and the optional CUDA-event timing (see nezha_profile_*).
enum KernelClass : int {
  kcGemm = 0, kcAttention, kcSelect, kcNorm, kcRope, kcEmbed, kcSwiglu, kcDraftGlue, kcNodes, kcAccept, kcHash, kcMisc,
  kcCount
};
static_assert(kcCount <= NEZHA_PROFILE_CLASSES, "profile classes");
// Wrap the launch(es) of one kernel class: counts them and, when profiling is on, brackets them with events.
struct LaunchScope {
  LaunchScope(int cls, cudaStream_t st, int n_launches = 1);
  ~LaunchScope();
  int cls; cudaStream_t st; int slot;
};

// --------------------------------------------------------------------------------------------------
// programmatic dependent launch: the kernels of the decode path are launched so that a kernel may be scheduled, and
// run the part of its prologue that touches no global memory, while its predecessor in the stream is still finishing
// --------------------------------------------------------------------------------------------------
// EVERY thread block of a kernel launched with launch_pdl must execute pdl_wait() before it touches anything that the
// preceding grid writes (or writes what that one reads), and before it exits (a block that exits without waiting lets the
// grid "complete" while its predecessor is still running, and the grid after it would then start too early).  What is older
// than the preceding grid may be read before, past the L1 (__ldcg, TMA): pdl_launch() always comes behind pdl_wait(), so when
// a block starts, all grids but that one are complete.  pdl_wait() returns once the preceding grid has
// completed and its writes are visible; pdl_launch() lets the following grid start being scheduled.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

bool pdl_enabled();     // false when NEZHA_NO_PDL is set: plain stream-ordered launches

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// --------------------------------------------------------------------------------------------------
// small device helpers
// --------------------------------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// --------------------------------------------------------------------------------------------------
// hash set (Eq. 5): open addressing over 32-byte buckets (one sector), linear probing over buckets
// --------------------------------------------------------------------------------------------------
// Two slot widths.  A code space of at most 2^32 tuples (every configured workload: 256^4, 512^3, 32^3) is stored NARROW:
// the key is sent through a bijection of the 32-bit integers and the slot holds the 32-bit image, so that a bucket has
// eight slots and the table half the bytes at the same number of slots -- a random probe of a table beyond the L2 costs a
// 64-byte DRAM access whatever it reads, so bytes of table are what a probe pays for (10M items at load factor 0.5: 160 MB
// -> 80 MB; the probe kernel's figures stand at hs_probe_kernel).  Larger spaces hold the 64-bit keys themselves, four per
// bucket.  The empty slot is all ones in both: no packed key in the wide form; in the narrow form one key may map to it,
// whose membership is a word of its own behind the buckets.
struct HashSetView {
  unsigned long long* slots;       // n_buckets buckets of kBucketBytes (+ one more that holds the special word, narrow form)
  unsigned long long n_buckets;    // narrow: below 2^31
  int narrow;
};

// 64-bit finalizer (the published murmur3 fmix64 constants), then multiply-shift range reduction so that
// any bucket count works (no power-of-two requirement).
__device__ __forceinline__ unsigned long long hs_mix(unsigned long long k) {
  k ^= k >> 33; k *= 0xff51afd7ed558ccdull; k ^= k >> 33; k *= 0xc4ceb9fe1a85ec53ull; k ^= k >> 33;
  return k;
}
__device__ __forceinline__ unsigned long long hs_bucket(unsigned long long key, unsigned long long n_buckets) {
  return __umul64hi(hs_mix(key), n_buckets);
}
// The 32-bit finalizer of the same family (fmix32): a bijection (xor-shifts and odd multipliers).
__device__ __forceinline__ unsigned hs_mix32(unsigned k) {
  k ^= k >> 16; k *= 0x85ebca6bu; k ^= k >> 13; k *= 0xc2b2ae35u; k ^= k >> 16;
  return k;
}
__device__ __forceinline__ const unsigned* hs_special(const HashSetView& hs) {
  return reinterpret_cast<const unsigned*>(hs.slots) + hs.n_buckets * (kBucketBytes / 4);
}

struct __align__(32) Bucket { unsigned w[8]; };          // one bucket, narrow slots or the halves of wide ones
__device__ __forceinline__ Bucket ld_bucket(const unsigned long long* slots, unsigned long long b) {
  Bucket r;                                              // one 32-byte request
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
      : "l"(slots + b * (kBucketBytes / 8)));
  return r;
}
// What a key is compared with: both halves of a wide slot, or (narrow) the image in every half.
struct SlotValue { unsigned lo, hi; };
template <bool NARROW> __device__ __forceinline__ SlotValue slot_value(unsigned long long key) {
  if constexpr (NARROW) { const unsigned m = hs_mix32((unsigned)key); return SlotValue{m, m}; }
  return SlotValue{(unsigned)key, (unsigned)(key >> 32)};
}
// What a bucket says about a key: 1 = it is here, 0 = it is nowhere (a free slot ends its walk), -1 = look further.
template <bool NARROW> __device__ __forceinline__ int bucket_verdict(const Bucket& k, SlotValue v) {
  bool hit = false, open = false;
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    const bool e0 = k.w[i] == v.lo, e1 = k.w[i + 1] == v.hi, o0 = k.w[i] == ~0u, o1 = k.w[i + 1] == ~0u;
    hit |= NARROW ? (e0 || e1) : (e0 && e1);
    open |= NARROW ? (o0 || o1) : (o0 && o1);
  }
  return hit ? 1 : open ? 0 : -1;
}
template <bool NARROW> __device__ __forceinline__ unsigned long long home_bucket(const HashSetView& hs, unsigned long long key) {
  if constexpr (NARROW) return __umulhi(hs_mix32((unsigned)key), (unsigned)hs.n_buckets);
  return hs_bucket(key, hs.n_buckets);
}
// The walk on from a home bucket that is full without holding the key: rare at the load factors in use.
template <bool NARROW>
__device__ __forceinline__ bool hs_walk_on(unsigned long long* slots, unsigned long long n_buckets, unsigned long long b,
                                               SlotValue v) {
  const HashSetView hs{slots, n_buckets, NARROW};
  for (int step = 1; step < kMaxProbeBuckets; ++step) {
    if (++b == n_buckets) b = 0;
    const int verdict = bucket_verdict<NARROW>(ld_bucket(hs.slots, b), v);
    if (verdict >= 0) return verdict > 0;
  }
  return false;
}

// Membership of N keys per thread with the memory round trips overlapped: the home buckets of all keys are loaded first
// (independent loads).
template <bool NARROW, int N>
__device__ __forceinline__ void hs_contains_form(const HashSetView& hs, const unsigned long long* keys, const bool* want,
                                                 bool* found) {
  Bucket k[N];
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (want[j]) k[j] = ld_bucket(hs.slots, home_bucket<NARROW>(hs, keys[j]));
#pragma unroll
  for (int j = 0; j < N; ++j) {
    found[j] = false;
    // outside the code space (narrow), or the free slots' value (wide): no member
    if (!want[j] || (NARROW ? keys[j] >> 32 != 0ull : keys[j] == kEmptyKey)) continue;
    const SlotValue v = slot_value<NARROW>(keys[j]);
    if (NARROW && v.lo == ~0u) { found[j] = __ldg(hs_special(hs)) != 0u; continue; }
    const int verdict = bucket_verdict<NARROW>(k[j], v);
    found[j] = verdict >= 0 ? verdict > 0 : hs_walk_on<NARROW>(hs.slots, hs.n_buckets, home_bucket<NARROW>(hs, keys[j]), v);
  }
}
// One key, either form.
__device__ __forceinline__ bool hs_contains_thread(const HashSetView& hs, unsigned long long key) {
  const bool want[1] = {true};
  bool found[1];
  if (hs.narrow) hs_contains_form<true, 1>(hs, &key, want, found);
  else hs_contains_form<false, 1>(hs, &key, want, found);
  return found[0];
}

// --------------------------------------------------------------------------------------------------
// prefix map: the same set V, regrouped as (prefix of n codes) -> bit set of the codes that may follow it
// --------------------------------------------------------------------------------------------------
// For every n in [0, L): the distinct n-code prefixes of the valid IDs, each with the bit set of the level-(n+1) codes t
// such that some valid ID begins with (prefix, t).  For n = L - 1 that is Eq. 5 itself for all T_L extensions of a beam in
// one look-up -- the same answers as T_L hash probes, bit for bit; for n < L - 1 it answers "does any valid ID begin with
// these codes?", the validity filter at the earlier levels.  One table region per n (so a key needs no level tag), in one of
// two forms, whichever takes fewer bytes for that n (launch-time constant, chosen where the arena is laid out):
//   direct   the bit sets of all prod T[:n] possible prefixes, indexed by the prefix key.  The short prefixes always, and
//            the longest ones of a catalogue that is dense in its prefix space (10M items over 256^3 prefixes: 537 MB
//            against 1.28 GB hashed, and an insertion is one atomic with no slot to find first)
//   hashed   open addressing with linear probing over slots of `stride` words: word 0 = prefix key + 1 (0 = empty), words
//            1.. = the bit set (1M items over 256^3 prefixes: 128 MB)
struct PrefixMapView {
  unsigned long long* slots;       // all regions, n_words words
  unsigned long long n_words;
  int stride, set_words;           // words per slot (a power of two >= 1 + set_words); words per bit set, ceil(max T / 64)
  unsigned long long level_off[kMaxLevels];     // first word of the region of prefixes with n codes
  unsigned long long level_slots[kMaxLevels];   // its slot count; 0 = direct
  unsigned long long level_keys[kMaxLevels];    // direct: the prefixes it has bit sets for
};
// The bit set of a prefix of n codes, or null (an empty set counts as none) if no valid ID begins with it.  Every lane of a
// warp may call this with the same key (the loads are then broadcasts).
__device__ __forceinline__ const unsigned long long* pm_find(const PrefixMapView& pm, int n, unsigned long long prefix_key) {
  const unsigned long long ns = pm.level_slots[n];
  const unsigned long long* region = pm.slots + pm.level_off[n];
  // (nezha_select takes a caller's codes as they are: a key beyond the code space begins no valid ID)
  if (ns == 0) return prefix_key < pm.level_keys[n] ? region + prefix_key * pm.set_words : nullptr;
  unsigned long long s = __umul64hi(hs_mix(prefix_key), ns);
  for (int step = 0; step < kMaxProbeBuckets; ++step) {
    const unsigned long long* slot = region + s * pm.stride;
    const unsigned long long k = __ldg(slot);
    if (k == prefix_key + 1) return slot + 1;
    if (k == 0ull) return nullptr;
    if (++s == ns) s = 0;
  }
  return nullptr;
}
__device__ __forceinline__ bool pm_test(const unsigned long long* bits, int t) {
  return bits != nullptr && ((__ldg(bits + (t >> 6)) >> (t & 63)) & 1ull);
}

// Plan and scratch of a build by parts (launch_set_build).  The items are dealt out twice: by runs of 2^shift prefixes of the
// prefix map's longest region, and by runs of 2^shift buckets of the hash set.
constexpr int kBuildBlocks = 148;         // blocks that share the catalogue out (one per SM of a B200; the scratch is laid out for them)
constexpr int kBuildMaxParts = 8192;
struct BuildDeal {
  int parts, shift;
  unsigned* count;                 // [parts + 1] keys of each part, then their exclusive sums
  unsigned* offset;                // [kBuildBlocks][parts] where a block's keys of a part start within the part
};
struct BuildScratch {
  int on;                          // 0: no build by parts
  BuildDeal by_prefix, by_bucket;
  unsigned* keys;                  // [n] the packed keys, part after part, of one deal after the other
  unsigned* n_valid;               // [kBuildBlocks] keys a block has packed
  unsigned* any;                   // [by_prefix.parts << shift] bits: which prefixes some item begins with
  unsigned* n_over;                // [by_bucket.parts] keys that ran over the end of a part (left at the part's start in keys)
};

// --------------------------------------------------------------------------------------------------
// model / engine description shared by the host code and the kernels
// --------------------------------------------------------------------------------------------------
struct LevelInfo {
  int L;
  int T[kMaxLevels];
  int off[kMaxLevels];             // vocabulary offset of each level's codes
  unsigned long long mult[kMaxLevels];   // Eq. 4 positional multipliers
  int vocab_codes;                 // sum(T)
};

// --------------------------------------------------------------------------------------------------
// GEMM:  C[M,N] (op)= A[M,K] * W[N,K]^T   (both operands K-major)
// --------------------------------------------------------------------------------------------------
enum GemmEpilogue : int {
  kEpiStoreAct = 0,     // C (activation type) = acc
  kEpiStoreF32 = 1,     // C (float) = acc
  kEpiAddF32 = 2,       // C (float) += acc                    (residual stream)
  kEpiBiasTanhF32 = 3,  // C (float) = tanh(acc + bias[n])     (Eq. 3)
  // ---- fused epilogues of the tensor-core kernel only -------------------------------------------------------
  kEpiSwiGLU = 4,       // weight rows interleaved (gate, gate, up, up per 4 columns): C (act)[m, n/2] = silu(gate) * up
  kEpiAddNorm = 5,      // C (float) += acc; xg (act)[m, n] = C * gain[n]; ss_out[n / 32][m] = sum of C^2 over the 32 columns
  kEpiRopeKV = 6        // fused QKV projection: rotary embedding on q and k, q to C, k and v to the KV cache
};

// Extras of the fused epilogues.  RMSNorm is split around the GEMMs: the producer of the residual stream
// (kEpiAddNorm) leaves x * gain as the next GEMM's A operand and partial sums of x^2 per 32 columns; the consumer GEMM
// multiplies its accumulator rows by rsqrt(mean(x^2) + eps), summing the partials in a fixed order.
struct GemmFuse {
  const float* ss_in; int ss_in_parts; long long ss_ld; float inv_dim, eps;   // row scale of the A operand (or null)
  float* ss_out;                     // [N / 32][ss_ld]
  void* xg; const void* gain;        // kEpiAddNorm: next A operand [M, N] (activation type) and its norm gain [N]
  // kEpiRopeKV: weight rows of every q / k head permuted so that every 4 consecutive columns hold two rotary pairs
  const int* tok_pos; const long long* kv_dst; long long kv_head_stride;
  void* k_cache; void* v_cache; const float* cos_tab; const float* sin_tab;
  int Hq, Hkv, hd;
};

constexpr int kSkinnyRows = 128;         // engines whose passes have at most this many rows stream every product's weights
constexpr int kSkinnyClassRows = 640;    // and at most this many: the products for which it pays (gemm_skinny_applies)

struct GemmArgs {
  const void* A; long long lda;
  const void* W; long long ldw;
  void* C; long long ldc;
  int M;                 // upper bound of rows (grid is sized for it)
  const int* M_dev;      // optional: actual row count on the device (<= M); rows beyond are skipped
  int N, K;
  int epilogue;
  const float* bias;
  int* status;           // device status word (bounded waits report here)
  GemmFuse f;            // zero-initialised unless a fused epilogue is asked for
  int M_expected;        // 0, or the row count the caller expects on the device (<= M): only shapes the tiling
  // Row class, or 0: the most rows that any launch of the caller's family may have (at most kSkinnyClassRows).  The product
  // may then run as the weight-streaming kernel (weights as the 128-row MMA operand, the rows as its N, the K range split
  // over the CTAs of a cluster), by a rule on (N, K), the class and the device only.  Its summation order differs from the
  // other kernels': a caller that needs the same bits from two launches gives both the same class.  W must be constant
  // data (it is read before the launch's dependency on its predecessor is resolved).
  int skinny;
  // Optional, and only a hint (the weight-streaming kernel heeds it, the others do not): constant data that the launch after
  // this one starts with, asked for into L2 while this launch waits for its predecessor.  16-byte aligned, a multiple of 16.
  const void* next_w; long long next_w_bytes;
  int early;             // W is constant and M_dev older than the launch before this one: both may be read while that one still runs
};

void launch_gemm_simt(const GemmArgs& a, bool bf16, cudaStream_t st);

// --------------------------------------------------------------------------------------------------
// element-wise / glue kernels
// --------------------------------------------------------------------------------------------------
void launch_embed(const void* table, bool bf16, const int* tokens, int M, const int* M_dev, int d, float* resid,
                  cudaStream_t st);
void launch_embed_norm(const void* table, const int* tokens, int M, const int* M_dev, int d, float* resid,
                       const void* gain, void* xg, float* ss, cudaStream_t st);
void launch_permute_rotary_rows(const void* src, void* dst, int rows, int hd, int cols, cudaStream_t st);
void launch_interleave_gate_up(const void* gate, const void* up, void* dst, int F, int cols, cudaStream_t st);
void launch_rmsnorm(const float* x, long long x_stride, const int* row_index, const void* gain, bool bf16, void* out,
                    float* out_f32, int M, const int* M_dev, int d, float eps, cudaStream_t st);

struct RopeAppendArgs {
  void* qkv;                       // [M, (Hq + 2 Hkv) * hd], activation type; q and k rotated in place
  const int* tok_pos;              // [M] rotary position
  const long long* kv_dst;         // [M] element offset of the token's K (and V) row group in the layer's cache:
                                   //     token's head h row starts at kv_dst[i] + h * kv_head_stride
  long long kv_head_stride;
  void* k_cache; void* v_cache;    // layer base pointers
  const float* cos_tab; const float* sin_tab;   // [positions, hd/2]
  int M; const int* M_dev;
  int Hq, Hkv, hd;
};
void launch_rope_append(const RopeAppendArgs& a, bool bf16, cudaStream_t st);
// fp32: C = RMSNorm(A, gain) W^T with, where `rope` is given, what launch_rope_append does (C = its qkv, of which only q is written) or,
// `swiglu`, C [M, N / 2] = what launch_swiglu makes of the product; else the product as it is.  Where norm_gemm_rows_applies.
bool norm_gemm_rows_applies(int M, int N, int K, const void* A, long long lda, const void* W, const void* gain);
void launch_norm_gemm_rows(const GemmArgs& a, const void* gain, float eps, const RopeAppendArgs* rope, bool swiglu, cudaStream_t st);
void launch_swiglu(const void* gu, void* act, int M, const int* M_dev, int F, bool bf16, cudaStream_t st);

// --------------------------------------------------------------------------------------------------
// attention over (context KV prefix) + (a few extra KV rows per token)
// --------------------------------------------------------------------------------------------------
struct AttnArgs {
  const void* q; long long q_stride;        // token i, head h at q + i*q_stride + h*hd
  void* out; long long out_stride;          // [M, Hq*hd]
  const void* k_ctx; const void* v_ctx;     // layer base of the context cache [rows][Hkv][S][hd]
  long long ctx_row_stride, ctx_head_stride;// element strides (row = request, head = kv head)
  const void* k_ext; const void* v_ext;     // layer base of the draft-token cache
  long long ext_head_stride;                // element stride between kv heads inside one extra entry
  const int* tok_row;                       // [M] request (cache row) of the token
  const int* tok_ctx_len;                   // [M] number of context positions visible
  const long long* tok_ext;                 // [M, n_ext_max] element offsets of extra KV entries, -1 = unused
  int n_ext_max;
  int M; const int* M_dev;
  int Hq, Hkv, hd;
  float scale;
  // grouping of the token list by request (tokens of a request are contiguous), for the tensor-core kernel
  const int* row_start; const int* row_count;   // [n_rows] first token / token count of each request in this pass
  const int4* req_info;                         // [n_rows] {first token, token count, cache row, context length visible to
                                                //  every token of the request, or -1: token j of the request sees j + 1}
  int n_rows, max_tokens_per_row;
  int split_max;                                // attention_split_max of the positions that a token may see
  int rows_expected;                            // 0, or the query rows per (request, kv head) the caller expects: tiling only
  // What the choice among kernels of different summation orders goes by: the query rows per (request, kv head) of one level's
  // beams, and of a whole draft tree (a prompt pass: both the longest prompt's).  Functions of the call's arguments alone, the
  // same in every round and mode, unlike rows_expected, which earlier calls leave behind: a repeated call returns the same
  // bits, and what one mode selects another verifies on the same sums.
  int rule_rows, rule_rows_most;
  long long ctx_rows_total;                     // requests * kv heads * positions of the layer's context cache
  // the draft-token cache seen as positions: a request owns ext_positions consecutive positions (level-major, then beam
  // slot), ext_pos_stride elements apart (all KV heads of a position are adjacent), ext_req_stride elements per request
  int ext_positions; long long ext_pos_stride, ext_req_stride, ext_rows_total;
  int* status;
};
void launch_attention_simt(const AttnArgs& a, bool bf16, cudaStream_t st);

}  // namespace nz
