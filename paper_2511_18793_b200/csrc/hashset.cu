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
template <typename Slot>
__device__ __forceinline__ int hs_insert_slot(unsigned long long* slots, unsigned long long n_buckets, unsigned long long b, Slot val) {
  constexpr int kSlots = kBucketBytes / sizeof(Slot);
  constexpr Slot kFree = ~(Slot)0;
  for (int step = 0; step < kMaxProbeBuckets; ++step) {
    Slot* bucket = reinterpret_cast<Slot*>(slots) + b * kSlots;
    for (int s = 0; s < kSlots; ++s) {
      Slot cur = *reinterpret_cast<volatile Slot*>(bucket + s);
      if (cur == kFree) {
        cur = atomicCAS(bucket + s, kFree, val);
        if (cur == kFree) return 1;
      }
      if (cur == val) return 0;
    }
    if (++b == n_buckets) b = 0;
  }
  return -1;
}

__global__ void hs_insert_kernel(LevelInfo li, HashSetView hs, const int* __restrict__ codes, unsigned long long n,
                                 unsigned long long* n_unique, int* status) {
  unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  bool inserted = false;
  if (i < n) {
    int c[kMaxLevels];
    load_codes<false>(codes, i, li.L, c);
    const unsigned long long key = pack_checked(li, c);
    if (key == kEmptyKey) {
      atomicOr(status, kStBadCode);
    } else {
      int r;
      const unsigned m = hs_mix32((unsigned)key);
      if (!hs.narrow) r = hs_insert_slot<unsigned long long>(hs.slots, hs.n_buckets, hs_bucket(key, hs.n_buckets), key);
      else if (m != ~0u) r = hs_insert_slot<unsigned>(hs.slots, hs.n_buckets, __umulhi(m, (unsigned)hs.n_buckets), m);
      else r = atomicExch(const_cast<unsigned*>(hs_special(hs)), 1u) == 0u ? 1 : 0;
      if (r < 0) atomicOr(status, kStHashFull);
      inserted = r > 0;
    }
  }
  unsigned m = __ballot_sync(0xffffffffu, inserted);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(n_unique, (unsigned long long)__popc(m));
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

// One thread per item: for every n in [0, L) it claims (or finds) the slot of the item's n-code prefix in region n and sets
// the bit of the item's next code.  The bit is tested first: the few prefixes at the top of the tree are shared by
// millions of items, whose atomics on the same word would otherwise serialise.
__global__ void pm_insert_kernel(LevelInfo li, PrefixMapView pm, const int* __restrict__ codes, unsigned long long n, int* status) {
  const unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int c[kMaxLevels];
  for (int l = 0; l < li.L; ++l) {
    c[l] = codes[i * li.L + l];
    if (c[l] < 0 || c[l] >= li.T[l]) return;        // hs_insert_kernel has reported it
  }
  unsigned long long p = 0;
  for (int lv = 0; lv < li.L; ++lv) {               // prefix of lv codes, next code c[lv]
    if (lv > 0) p += (unsigned long long)c[lv - 1] * li.mult[lv - 1];
    const int t = c[lv];
    const unsigned long long ns = pm.level_slots[lv];
    unsigned long long* region = pm.slots + pm.level_off[lv] * pm.stride;
    unsigned long long s = __umul64hi(hs_mix(p), ns);
    bool done = false;
    for (int step = 0; step < kMaxProbeBuckets && !done; ++step) {
      unsigned long long* slot = region + s * pm.stride;
      unsigned long long cur = *reinterpret_cast<volatile unsigned long long*>(slot);
      if (cur == 0ull) cur = atomicCAS(slot, 0ull, p + 1);
      if (cur == 0ull || cur == p + 1) {
        unsigned long long* word = slot + 1 + (t >> 6);
        const unsigned long long bit = 1ull << (t & 63);
        if (!(*reinterpret_cast<volatile unsigned long long*>(word) & bit)) atomicOr(word, bit);
        done = true;
      }
      if (++s == ns) s = 0;
    }
    if (!done) { atomicOr(status, kStHashFull); return; }
  }
}

void launch_pm_build(const LevelInfo& li, PrefixMapView pm, const int* codes, unsigned long long n, int* status, cudaStream_t st) {
  if (!pm.slots) return;
  cudaMemsetAsync(pm.slots, 0, (size_t)pm.n_slots * pm.stride * sizeof(unsigned long long), st);
  if (!n) return;
  LaunchScope ls(kcHash, st);
  pm_insert_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(li, pm, codes, n, status);
}

void launch_hs_clear(HashSetView hs, cudaStream_t st) {
  cudaMemsetAsync(hs.slots, 0xff, (size_t)hs.n_buckets * kBucketBytes, st);
  cudaMemsetAsync(hs.slots + hs.n_buckets * (kBucketBytes / 8), 0, kBucketBytes, st);      // the special word (HashSetView)
}
void launch_hs_pack(const LevelInfo& li, const int* codes, unsigned long long n, unsigned long long* keys, int* status,
                    cudaStream_t st) {
  if (!n) return;
  LaunchScope ls(kcHash, st);
  const unsigned grid = (unsigned)((n + 511) / 512);
  if (codes_vec(li, codes)) hs_pack_kernel<true><<<grid, 256, 0, st>>>(li, codes, n, keys, status);
  else hs_pack_kernel<false><<<grid, 256, 0, st>>>(li, codes, n, keys, status);
}
void launch_hs_insert(const LevelInfo& li, HashSetView hs, const int* codes, unsigned long long n,
                      unsigned long long* n_unique, int* status, cudaStream_t st) {
  if (!n) return;
  LaunchScope ls(kcHash, st);
  hs_insert_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(li, hs, codes, n, n_unique, status);
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
