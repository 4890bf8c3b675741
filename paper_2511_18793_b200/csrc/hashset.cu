// Eq. 4 (mixed-radix packing) and Eq. 5 (the set V of valid IDs) on the GPU.
//
// V is an open-addressing hash set of packed keys in buckets of one 32-byte sector (HashSetView: the two slot widths).  A
// key hashes to a bucket and probes linearly over buckets.  Insertion takes the first empty slot of the first non-full
// bucket on its probe path, so a lookup can stop at the first bucket that still has an empty slot.  A lookup is one
// thread reading whole buckets (one 32-byte load); stand-alone lookups take two keys per thread so that both sectors are
// in flight together.  All walks are bounded by kMaxProbeBuckets.
#include "common.cuh"

namespace nz {

// The L codes of item i; VEC: rows of 4 or 8 codes on 16-byte boundaries are fetched whole (with one load per code a warp
// spreads every load over L times the lines).
template <bool VEC>
__device__ __forceinline__ void load_codes(const int* __restrict__ codes, unsigned long long i, int L, int* c) {
  if constexpr (VEC) {
#pragma unroll
    for (int l = 0; l < kMaxLevels; l += 4)
      if (l < L) {
        const int4 v = __ldcs(reinterpret_cast<const int4*>(codes + i * L + l));
        c[l] = v.x; c[l + 1] = v.y; c[l + 2] = v.z; c[l + 3] = v.w;
      }
  } else {
#pragma unroll
    for (int l = 0; l < kMaxLevels; ++l)
      if (l < L) c[l] = __ldg(codes + i * L + l);
  }
}
inline bool codes_vec(const LevelInfo& li, const int* codes) { return li.L % 4 == 0 && ((uintptr_t)codes & 15) == 0; }

// Eq. 4; kEmptyKey for a tuple with a code outside its codebook.
__device__ __forceinline__ unsigned long long pack_checked(const LevelInfo& li, const int* c) {
  unsigned long long k = 0;
  bool bad = false;
#pragma unroll
  for (int l = 0; l < kMaxLevels; ++l)
    if (l < li.L) {
      bad |= (unsigned)c[l] >= (unsigned)li.T[l];
      k += (unsigned long long)c[l] * li.mult[l];
    }
  return bad ? kEmptyKey : k;
}

// Streaming: 16 bytes in, 8 out for L = 4.  2^24 tuples: 99 us with one item per thread and a load per code, 67 us
// (6.0 TB/s, 0.92 of the copy bandwidth) with two items per thread and whole rows.
template <bool VEC>
__global__ void __launch_bounds__(256) hs_pack_kernel(LevelInfo li, const int* __restrict__ codes, unsigned long long n,
                                                      unsigned long long* __restrict__ keys, int* status) {
  const unsigned long long base = blockIdx.x * 512ull + threadIdx.x;
  int c[2][kMaxLevels];
#pragma unroll
  for (int j = 0; j < 2; ++j)
    if (base + 256 * j < n) load_codes<VEC>(codes, base + 256 * j, li.L, c[j]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (base + 256 * j >= n) break;
    const unsigned long long k = pack_checked(li, c[j]);
    if (k == kEmptyKey) atomicOr(status, kStBadCode);
    keys[base + 256 * j] = k;
  }
}

// Claims a slot for `val` in the bucket walk that starts at bucket b: 1 = inserted, 0 = already there, -1 = table full.
// The bucket is looked at with one plain load.  What it shows may be out of date, but only in one direction -- a slot that
// looks free may have been taken since -- and the compare-and-swap says by whom.  (A compare-and-swap without a look, at a
// slot the hash names: slower, 1,004 us against 778 for 10M items, because some lane of a warp always has to go on.)
template <typename Slot>
__device__ __forceinline__ int hs_insert_slot(unsigned long long* slots, unsigned long long n_buckets, unsigned long long b, Slot val) {
  constexpr int kSlots = kBucketBytes / sizeof(Slot);
  constexpr Slot kFree = ~(Slot)0;
  for (int step = 0; step < kMaxProbeBuckets; ++step) {
    Slot* bucket = reinterpret_cast<Slot*>(slots) + b * kSlots;
    union { unsigned w[8]; Slot s[kSlots]; } k;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(k.w[0]), "=r"(k.w[1]), "=r"(k.w[2]), "=r"(k.w[3]), "=r"(k.w[4]), "=r"(k.w[5]), "=r"(k.w[6]), "=r"(k.w[7])
                 : "l"(bucket) : "memory");
    int first_free = kSlots;
#pragma unroll
    for (int s = kSlots - 1; s >= 0; --s) {
      if (k.s[s] == val) return 0;
      if (k.s[s] == kFree) first_free = s;
    }
    for (int s = first_free; s < kSlots; ++s) {
      const Slot cur = atomicCAS(bucket + s, kFree, val);
      if (cur == kFree) return 1;
      if (cur == val) return 0;
    }
    if (++b == n_buckets) b = 0;
  }
  return -1;
}

// Sets the bit of code t behind a prefix of n codes: 1 = the prefix may not have been there before, 0 = it was, -1 = full.
// (`fresh`: the bit is known to be clear.  Otherwise it is tested first, with a plain cached load -- a stale answer costs
// an atomic, no more: the few prefixes at the top of the tree are shared by millions of items.)
__device__ __forceinline__ int pm_add(const PrefixMapView& pm, int n, unsigned long long p, int t, bool fresh) {
  const unsigned long long ns = pm.level_slots[n], bit = 1ull << (t & 63);
  unsigned long long* region = pm.slots + pm.level_off[n];
  if (ns == 0) {
    unsigned long long* word = region + p * pm.set_words + (t >> 6);
    if (!fresh && (*word & bit)) return 0;
    return atomicOr(word, bit) == 0ull ? 1 : 0;          // (a prefix of several words may say so once per word)
  }
  unsigned long long s = __umul64hi(hs_mix(p), ns);
  for (int step = 0; step < kMaxProbeBuckets; ++step) {
    unsigned long long* slot = region + s * pm.stride;
    unsigned long long cur = *slot;
    bool claimed = false;
    if (cur == 0ull) { cur = atomicCAS(slot, 0ull, p + 1); claimed = cur == 0ull; }
    if (claimed || cur == p + 1) {
      unsigned long long* word = slot + 1 + (t >> 6);
      if (fresh || !(*word & bit)) atomicOr(word, bit);
      return claimed ? 1 : 0;
    }
    if (++s == ns) s = 0;
  }
  return -1;
}

// The hash set and the prefix map in one pass over the catalogue.  An item that is in the set already is done.  A new one
// sets its bit behind its L - 1 codes, and only where that prefix was not there yet does it go on to the next shorter one:
// whoever brought a prefix has entered it everywhere above, so almost every item ends after two or three random accesses
// (an insertion that walks all L prefixes per item was bound by the one cache line of the shortest).
// Bound by random atomics: measured alone 100 G/s on 80 MB, which L2 holds, 25 G/s on 537 MB, whatever their kind and
// whether or not their answer is used.  10M items: two kernels, every prefix of every item, hashed regions 1,540 us (and
// 229 us to clear them); this one 778 us (and 115).  Four items per thread in step: 1,657 us.
template <bool VEC, bool NARROW>
__global__ void __launch_bounds__(256) set_build_kernel(LevelInfo li, HashSetView hs, PrefixMapView pm, const int* __restrict__ codes,
                                                        unsigned long long n, unsigned long long* n_unique, int* status) {
  int inserted = 0;
  for (unsigned long long i = blockIdx.x * 256ull + threadIdx.x; i < n; i += gridDim.x * 256ull) {
    int c[kMaxLevels];
    load_codes<VEC>(codes, i, li.L, c);
    const unsigned long long key = pack_checked(li, c);
    if (key == kEmptyKey) { atomicOr(status, kStBadCode); continue; }
    int r;
    if constexpr (NARROW) {
      const unsigned m = hs_mix32((unsigned)key);
      if (m != ~0u) r = hs_insert_slot<unsigned>(hs.slots, hs.n_buckets, __umulhi(m, (unsigned)hs.n_buckets), m);
      else r = atomicExch(const_cast<unsigned*>(hs_special(hs)), 1u) == 0u ? 1 : 0;
    } else {
      r = hs_insert_slot<unsigned long long>(hs.slots, hs.n_buckets, hs_bucket(key, hs.n_buckets), key);
    }
    if (r > 0) {
      ++inserted;
      unsigned long long p = key;
      bool fresh = true;
#pragma unroll
      for (int lv = kMaxLevels - 1; lv >= 0; --lv) {
        if (lv >= li.L || r <= 0) continue;
        p -= (unsigned long long)c[lv] * li.mult[lv];     // the prefix of lv codes
        r = pm_add(pm, lv, p, c[lv], fresh);
        fresh = false;
      }
    }
    if (r < 0) atomicOr(status, kStHashFull);
  }
  inserted = (int)__reduce_add_sync(0xffffffffu, (unsigned)inserted);
  __shared__ int part[8];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = inserted;
  __syncthreads();
  if (threadIdx.x == 0) {
    int sum = 0;
    for (int w = 0; w < 8; ++w) sum += part[w];
    if (sum) atomicAdd(n_unique, (unsigned long long)sum);
  }
}

// A thread answers kProbeKeysPerThread keys: it loads them (coalesced: thread t of the block takes keys t, t + 256, ...),
// asks for all their home buckets at once -- one 32-byte sector each, the only traffic that is not streaming -- and only
// then compares.  Bound by random sectors: L1 requests while the table is in L2 (one 32-byte load per bucket in place of
// two of 16), 64-byte DRAM accesses beyond it.  2^24 keys, half of them hits, wide slots and two loads -> narrow slots:
// 163 -> 91 us (1M items), 221 -> 101 us (10M items, table 160 -> 80 MB), 331 -> 258 us (33M items).  More keys per
// thread were slower when last measured (1, 2, 4, 8 keys: 106, 108, 85, 55 G probes/s on a table in L2).
constexpr int kProbeKeysPerThread = 2;
template <bool NARROW>
__global__ void __launch_bounds__(256) hs_probe_kernel(HashSetView hs, const unsigned long long* __restrict__ keys,
                                                       unsigned long long n, uint8_t* __restrict__ found) {
  const unsigned long long base = (unsigned long long)blockIdx.x * (256u * kProbeKeysPerThread) + threadIdx.x;
  unsigned long long k[kProbeKeysPerThread];
  bool want[kProbeKeysPerThread], hit[kProbeKeysPerThread];
#pragma unroll
  for (int j = 0; j < kProbeKeysPerThread; ++j) {
    const unsigned long long i = base + 256ull * j;
    want[j] = i < n;
    k[j] = want[j] ? __ldcs(keys + i) : 0ull;
    hit[j] = false;
  }
  hs_contains_form<NARROW, kProbeKeysPerThread>(hs, k, want, hit);
#pragma unroll
  for (int j = 0; j < kProbeKeysPerThread; ++j) {
    const unsigned long long i = base + 256ull * j;
    if (want[j]) found[i] = hit[j] ? 1 : 0;
  }
}

// Clears both tables and enters the n items; *n_unique = how many of them are distinct.
void launch_set_build(const LevelInfo& li, HashSetView hs, PrefixMapView pm, const int* codes, unsigned long long n,
                      unsigned long long* n_unique, int* status, int n_sm, cudaStream_t st) {
  cudaMemsetAsync(n_unique, 0, sizeof(unsigned long long), st);
  cudaMemsetAsync(hs.slots, 0xff, (size_t)hs.n_buckets * kBucketBytes, st);
  cudaMemsetAsync(hs.slots + hs.n_buckets * (kBucketBytes / 8), 0, kBucketBytes, st);      // the special word (HashSetView)
  cudaMemsetAsync(pm.slots, 0, (size_t)pm.n_words * sizeof(unsigned long long), st);
  if (!n) return;
  LaunchScope ls(kcHash, st);
  const unsigned long long blocks = (n + 255) / 256;
  const unsigned grid = (unsigned)(blocks < 8ull * n_sm ? blocks : 8ull * n_sm);
  auto go = [&](auto kernel) { kernel<<<grid, 256, 0, st>>>(li, hs, pm, codes, n, n_unique, status); };
  if (codes_vec(li, codes)) { if (hs.narrow) go(set_build_kernel<true, true>); else go(set_build_kernel<true, false>); }
  else { if (hs.narrow) go(set_build_kernel<false, true>); else go(set_build_kernel<false, false>); }
}
void launch_hs_pack(const LevelInfo& li, const int* codes, unsigned long long n, unsigned long long* keys, int* status,
                    cudaStream_t st) {
  if (!n) return;
  LaunchScope ls(kcHash, st);
  const unsigned grid = (unsigned)((n + 511) / 512);
  if (codes_vec(li, codes)) hs_pack_kernel<true><<<grid, 256, 0, st>>>(li, codes, n, keys, status);
  else hs_pack_kernel<false><<<grid, 256, 0, st>>>(li, codes, n, keys, status);
}
void launch_hs_probe(HashSetView hs, const unsigned long long* keys, unsigned long long n, uint8_t* found,
                     cudaStream_t st) {
  if (!n) return;
  const unsigned long long per_block = 256ull * kProbeKeysPerThread;
  LaunchScope ls(kcHash, st);
  const unsigned grid = (unsigned)((n + per_block - 1) / per_block);
  if (hs.narrow) hs_probe_kernel<true><<<grid, 256, 0, st>>>(hs, keys, n, found);
  else hs_probe_kernel<false><<<grid, 256, 0, st>>>(hs, keys, n, found);
}

}  // namespace nz
