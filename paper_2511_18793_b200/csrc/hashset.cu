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
template <typename Slot> struct SlotBucket {
  static constexpr int kSlots = kBucketBytes / sizeof(Slot);
  static constexpr Slot kFree = ~(Slot)0;
  union { unsigned w[8]; Slot s[kSlots]; };
  __device__ __forceinline__ void load(const Slot* bucket) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(bucket) : "memory");
  }
  __device__ __forceinline__ bool has(Slot val) const {
    bool hit = false;
#pragma unroll
    for (int i = 0; i < kSlots; ++i) hit |= s[i] == val;
    return hit;
  }
  __device__ __forceinline__ int first_free() const {
    int f = kSlots;
#pragma unroll
    for (int i = kSlots - 1; i >= 0; --i)
      if (s[i] == kFree) f = i;
    return f;
  }
};
template <typename Slot>
__device__ __forceinline__ int hs_insert_slot(unsigned long long* slots, unsigned long long n_buckets, unsigned long long b, Slot val) {
  using B = SlotBucket<Slot>;
  for (int step = 0; step < kMaxProbeBuckets; ++step) {
    Slot* bucket = reinterpret_cast<Slot*>(slots) + b * B::kSlots;
    B k;
    k.load(bucket);
    if (k.has(val)) return 0;
    for (int s = k.first_free(); s < B::kSlots; ++s) {
      const Slot cur = atomicCAS(bucket + s, B::kFree, val);
      if (cur == B::kFree) return 1;
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

template <bool NARROW>
__device__ __forceinline__ int hs_insert(const HashSetView& hs, unsigned long long key) {
  if constexpr (NARROW) {
    const unsigned m = hs_mix32((unsigned)key);
    if (m != ~0u) return hs_insert_slot<unsigned>(hs.slots, hs.n_buckets, __umulhi(m, (unsigned)hs.n_buckets), m);
    return atomicExch(const_cast<unsigned*>(hs_special(hs)), 1u) == 0u ? 1 : 0;
  } else {
    return hs_insert_slot<unsigned long long>(hs.slots, hs.n_buckets, hs_bucket(key, hs.n_buckets), key);
  }
}

// Adds a block's inserted items up (every thread of the block calls this once).
__device__ __forceinline__ void count_inserted(int inserted, unsigned long long* n_unique) {
  inserted = (int)__reduce_add_sync(0xffffffffu, (unsigned)inserted);
  __shared__ int part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = inserted;
  __syncthreads();
  if (threadIdx.x == 0) {
    int sum = 0;
    for (int w = 0; w < (int)blockDim.x >> 5; ++w) sum += part[w];
    if (sum) atomicAdd(n_unique, (unsigned long long)sum);
  }
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
    int r = hs_insert<NARROW>(hs, key);
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
  count_inserted(inserted, n_unique);
}

// ---- the same build by parts, for many items ---------------------------------------------------------------------------------
// Above, an item is a random access to a table that DRAM holds (bits; 10M items: 403 us of atomics on 537 MB) and two to one that
// the L2 holds (bucket, then slot; 254 us), behind a pass that clears both.  Here the items are dealt out to parts that a block's
// shared memory holds: by prefix, for the bits, and by bucket, for the hash set.  A block builds a part there and writes it
// once, which also replaces the clearing.
// 10M items over 256^4 codes, load factor 0.5, whole calls: 968 us above, 390 here, of which the bits take 86 (537 MB written; 82
// at the copy bandwidth), the slots 67, counting 58, the two deals 70 and 41, the rest launches.  30M: 2,907 -> 1,157.
// key / prefixes (the last code, at most 1,023) and the remainder.  Both roundings go down, and by less than 2^-10 of 1,024: the
// product's integer part is the quotient or one less.  (With the compiler's division the first deal of 10M items took 69 us, not 66.)
struct KeySplit {
  unsigned prefixes; float inv;     // inv: below 1 / prefixes
  __device__ __forceinline__ unsigned operator()(unsigned key, unsigned* prefix) const {
    unsigned t = __float2uint_rz(__fmul_rz(__uint2float_rz(key), inv));
    unsigned p = key - t * prefixes;
    if (p >= prefixes) { p -= prefixes; ++t; }
    *prefix = p;
    return t;
  }
};
struct DealPrefix {
  KeySplit split; int shift;
  __device__ __forceinline__ int operator()(unsigned key) const {
    unsigned p;
    split(key, &p);
    return (int)(p >> shift);
  }
};
struct DealBucket {
  unsigned n_buckets; int shift;
  __device__ __forceinline__ int operator()(unsigned key) const { return (int)(__umulhi(hs_mix32(key), n_buckets) >> shift); }
};

// The items in kBuildBlocks equal runs, one per block: packs a run's keys (left in keys[] at the run's start, without those
// with a bad code) and counts them by part, for both deals.  The block's place within each part is what the counter held before.
constexpr int kCountItems = 4, kCountRing = 2, kCountRingBytes = kCountRing * kCountItems * 1024 * 16;
template <bool VEC, bool RING>      // RING: VEC and four codes an item
__global__ void __launch_bounds__(1024) part_count_kernel(LevelInfo li, HashSetView hs, PrefixMapView pm, BuildScratch sc, DealBucket by_bucket,
                                                          const int* __restrict__ codes, unsigned n, unsigned run,
                                                          unsigned* __restrict__ keys, unsigned long long* n_unique, int* status) {
  extern __shared__ __align__(16) unsigned hist[];      // [by_prefix.parts], [by_bucket.parts], then (RING) kCountRing x kItems x 1024 items
  __shared__ unsigned n_keys;
  const int parts = sc.by_prefix.parts, both = parts + sc.by_bucket.parts;
  int4* ring = reinterpret_cast<int4*>(hist + (both + 3) / 4 * 4);
  for (int p = threadIdx.x; p < both; p += 1024) hist[p] = 0;
  if (threadIdx.x == 0) n_keys = 0;
  // what the kernels behind this one add to: the regions of the shorter prefixes, the special word, the number of items
  for (unsigned long long w = blockIdx.x * 1024ull + threadIdx.x; w < pm.level_off[li.L - 1]; w += kBuildBlocks * 1024ull) pm.slots[w] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) { *const_cast<unsigned*>(hs_special(hs)) = 0; *n_unique = 0; }
  __syncthreads();
  const unsigned lo = min(n, blockIdx.x * run), hi = min(n, lo + run);
  const int lane = threadIdx.x & 31;
  constexpr int kItems = kCountItems;                   // per thread and step
  // RING: a thread's items of the next steps are on their way into shared memory, read by nobody else (10M items: 66 -> 58 us, and as much
  // of the whole call as its runs differ by; 30M: the call 1,198 -> 1,152).  Rows of three codes are not copied so: their 12 bytes lie on no
  // 16-byte boundaries.
  auto ask = [&](unsigned i0, int slot) {
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const unsigned i = i0 + 1024 * j + threadIdx.x;
      if (i0 < hi && i < hi) {
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(ring + (slot * kItems + j) * 1024 + threadIdx.x);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at), "l"(codes + (unsigned long long)i * 4) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if constexpr (RING)
    for (int st = 0; st < kCountRing - 1; ++st) ask(lo + 1024 * kItems * st, st);
  int slot = 0;
  for (unsigned i0 = lo; i0 < hi; i0 += 1024 * kItems) {
    int c[kItems][RING ? 4 : kMaxLevels];
    if constexpr (RING) {
      ask(i0 + 1024 * kItems * (kCountRing - 1), (slot + kCountRing - 1) % kCountRing);
      asm volatile("cp.async.wait_group %0;" ::"n"(kCountRing - 1) : "memory");
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        const int4 v = ring[(slot * kItems + j) * 1024 + threadIdx.x];
        c[j][0] = v.x; c[j][1] = v.y; c[j][2] = v.z; c[j][3] = v.w;
      }
      slot = (slot + 1) % kCountRing;
    } else {
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        const unsigned i = i0 + 1024 * j + threadIdx.x;
        if (i < hi) load_codes<VEC>(codes, i, li.L, c[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const unsigned i = i0 + 1024 * j + threadIdx.x;
      unsigned prefix = 0, last = 0;
      bool ok = i < hi;
#pragma unroll
      for (int l = 0; l < (RING ? 4 : kMaxLevels); ++l)
        if (l < li.L && i < hi) {
          ok &= (unsigned)c[j][l] < (unsigned)li.T[l];
          const unsigned term = (unsigned)c[j][l] * (unsigned)li.mult[l];
          if (l == li.L - 1) last = term; else prefix += term;
        }
      if (i < hi && !ok) atomicOr(status, kStBadCode);
      const unsigned members = __ballot_sync(0xffffffffu, ok);
      unsigned at = 0;
      if (lane == 0 && members) at = atomicAdd(&n_keys, (unsigned)__popc(members));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (ok) {
        keys[lo + at + __popc(members & ((1u << lane) - 1))] = prefix + last;
        atomicAdd(&hist[prefix >> sc.by_prefix.shift], 1u);
        atomicAdd(&hist[parts + by_bucket(prefix + last)], 1u);
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) sc.n_valid[blockIdx.x] = n_keys;
  for (int p = threadIdx.x; p < both; p += 1024) {
    const BuildDeal& dl = p < parts ? sc.by_prefix : sc.by_bucket;
    const int q = p < parts ? p : p - parts;
    const unsigned h = hist[p];
    dl.offset[(size_t)blockIdx.x * dl.parts + q] = h ? atomicAdd(&dl.count[q], h) : 0u;
  }
}

// v[] of every thread of a block of 1024 (thread t: elements kEach t ..) becomes the exclusive prefix sums; returns what comes after
// the thread's elements.  tmp: 32 words of shared memory, free again after the next barrier.
template <int kEach>
__device__ __forceinline__ unsigned block_exclusive_sums(unsigned (&v)[kEach], unsigned* tmp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned sum = 0;
#pragma unroll
  for (int j = 0; j < kEach; ++j) sum += v[j];
  unsigned incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  const unsigned before = __reduce_add_sync(0xffffffffu, lane < warp ? tmp[lane] : 0u);
  unsigned start = before + incl - sum;
#pragma unroll
  for (int j = 0; j < kEach; ++j) { const unsigned x = v[j]; v[j] = start; start += x; }
  return start;
}

// The counts become the parts' starts (one block of 1024 threads per deal).
constexpr int kPartsEach = kBuildMaxParts / 1024;
__global__ void __launch_bounds__(1024) part_scan_kernel(BuildScratch sc) {
  __shared__ unsigned tmp[32];
  const BuildDeal& dl = blockIdx.x == 0 ? sc.by_prefix : sc.by_bucket;
  unsigned v[kPartsEach];
#pragma unroll
  for (int j = 0; j < kPartsEach; ++j) {
    const int p = threadIdx.x * kPartsEach + j;
    v[j] = p < dl.parts ? dl.count[p] : 0u;
  }
  const unsigned total = block_exclusive_sums(v, tmp);
#pragma unroll
  for (int j = 0; j < kPartsEach; ++j) {
    const int p = threadIdx.x * kPartsEach + j;
    if (p < dl.parts) dl.count[p] = v[j];
  }
  if (threadIdx.x == 1023) dl.count[dl.parts] = total;
}

// Deals a run's keys out to the parts, kDealKeys at a time: sorted by part in shared memory first, so that a part's keys go out
// as one piece.  (Each key stored by itself: 92 us for 10M keys and 8,192 parts, 110 G stores/s; so: 66, and 41 for 1,221 parts)
constexpr int kDealKeys = 32 << 10;
template <typename Deal>
__global__ void __launch_bounds__(1024) part_deal_kernel(BuildDeal dl, Deal part_of, const unsigned* __restrict__ n_valid, unsigned n,
                                                         unsigned run, const unsigned* __restrict__ keys, unsigned* __restrict__ out) {
  extern __shared__ unsigned sorted[];                  // [kDealKeys], then cursor[parts], base[parts]
  __shared__ unsigned tmp[32];
  unsigned *cursor = sorted + kDealKeys, *base = cursor + dl.parts;
  for (int p = threadIdx.x; p < dl.parts; p += 1024) {
    cursor[p] = 0;
    base[p] = dl.count[p] + dl.offset[(size_t)blockIdx.x * dl.parts + p];
  }
  const unsigned lo = min(n, blockIdx.x * run), hi = lo + n_valid[blockIdx.x];
  for (unsigned i0 = lo; i0 < hi; i0 += kDealKeys) {
    const unsigned cnt = min((unsigned)kDealKeys, hi - i0);
    // base + cursor = where the part's next key goes; the cursor starts again as a count
    __syncthreads();
    for (int p = threadIdx.x; p < dl.parts; p += 1024) { base[p] += cursor[p]; cursor[p] = 0; }
    __syncthreads();
#pragma unroll 4
    for (unsigned i = threadIdx.x; i < cnt; i += 1024) atomicAdd(&cursor[part_of(keys[i0 + i])], 1u);
    __syncthreads();
    unsigned v[kPartsEach];
#pragma unroll
    for (int j = 0; j < kPartsEach; ++j) {
      const int p = threadIdx.x * kPartsEach + j;
      v[j] = p < dl.parts ? cursor[p] : 0u;
    }
    block_exclusive_sums(v, tmp);
#pragma unroll
    for (int j = 0; j < kPartsEach; ++j) {
      const int p = threadIdx.x * kPartsEach + j;
      if (p < dl.parts) { cursor[p] = v[j]; base[p] -= v[j]; }
    }
    __syncthreads();
#pragma unroll 4
    for (unsigned i = threadIdx.x; i < cnt; i += 1024) {
      const unsigned k = keys[i0 + i];
      sorted[atomicAdd(&cursor[part_of(k)], 1u)] = k;
    }
    __syncthreads();
#pragma unroll 4
    for (unsigned i = threadIdx.x; i < cnt; i += 1024) {
      const unsigned k = sorted[i];
      out[base[part_of(k)] + i] = k;
    }
  }
}

// A copy from shared to global memory by the copy engine; one thread's, 16-byte aligned, a multiple of 16.  Every thread that has written
// the source fences before the barrier in front of it, and the source has to outlive it.
// STREAM: what is written is the first to leave the L2 again.
__device__ __forceinline__ void bulk_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
template <bool STREAM>
__device__ __forceinline__ void bulk_store(void* dst, const void* src, unsigned bytes) {
  const uint32_t at = (uint32_t)__cvta_generic_to_shared(src);
  if constexpr (STREAM) {
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(dst), "r"(at), "r"(bytes), "l"(policy) : "memory");
  } else {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(at), "r"(bytes) : "memory");
  }
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// One block per part of the prefix map's longest region: its bits, which of its prefixes begin an item, and how many items are
// distinct.
__global__ void __launch_bounds__(512, 3) part_bits_kernel(PrefixMapView pm, BuildScratch sc, int last, KeySplit split,
                                                           unsigned long long* n_unique) {
  extern __shared__ __align__(16) unsigned bits[];      // [2^shift][2 * set_words], then [2^shift / 32] for sc.any
  const int shift = sc.by_prefix.shift, row = 2 * pm.set_words, all = row << shift, any_words = 1 << (shift - 5);
  unsigned* any = bits + all;
  for (int w = threadIdx.x * 4; w < all; w += 512 * 4) *reinterpret_cast<uint4*>(bits + w) = make_uint4(0, 0, 0, 0);
  for (int w = threadIdx.x; w < any_words; w += 512) any[w] = 0;
  const unsigned begin = sc.by_prefix.count[blockIdx.x], end = sc.by_prefix.count[blockIdx.x + 1], p0 = (unsigned)blockIdx.x << shift;
  __syncthreads();
  int inserted = 0;
  for (unsigned i = begin + threadIdx.x; i < end; i += 512) {
    unsigned p;
    const unsigned t = split(sc.keys[i], &p), bit = 1u << (t & 31);
    p -= p0;
    unsigned* word = bits + p * row + (t >> 5);
    if (*(volatile unsigned*)word & bit) continue;       // (a repeated item; the popular ones are worth the look)
    const unsigned was = atomicOr(word, bit);
    if (was == 0) atomicOr(any + (p >> 5), 1u << (p & 31));
    inserted += !(was & bit);
  }
  bulk_fence();
  __syncthreads();
  const unsigned words = min(1u << shift, split.prefixes - p0) * pm.set_words;
  unsigned long long* out = pm.slots + pm.level_off[last] + (unsigned long long)p0 * pm.set_words;
  // One bulk copy out of shared memory, none of it through the threads' registers.  The region is larger than the L2, and what the next
  // kernels read -- the packed keys -- is in there: 10M items of 256^4 / 1,024^3 codes by the threads' streaming stores 122 / 91 us (and the
  // second deal 41 / 41), by a plain bulk copy 111 / 115 (51 / 49), by this one 86 / 83 (41 / 41).
  if (threadIdx.x == 0 && words >= 2) bulk_store<true>(out, bits, words / 2 * 16);
  if (threadIdx.x == 0 && (words & 1)) out[words - 1] = reinterpret_cast<const unsigned long long*>(bits)[words - 1];
  for (int w = threadIdx.x; w < any_words; w += 512) sc.any[(size_t)blockIdx.x * any_words + w] = any[w];
  count_inserted(inserted, n_unique);
  if (threadIdx.x == 0) bulk_wait();
}

// One block per part of the hash set: its buckets.  A key whose walk runs over the part's end goes back to the start of the
// part's keys, for part_over_kernel; those read so far are at least as many, hence the barrier between reading and writing.
__global__ void __launch_bounds__(512, 3) part_slots_kernel(HashSetView hs, BuildScratch sc) {
  using B = SlotBucket<unsigned>;
  extern __shared__ __align__(16) unsigned slots[];     // [2^shift][8]
  __shared__ unsigned n_over;
  const int shift = sc.by_bucket.shift;
  const unsigned b0 = (unsigned)blockIdx.x << shift, n_local = min(1u << shift, (unsigned)hs.n_buckets - b0);
  const unsigned begin = sc.by_bucket.count[blockIdx.x], end = sc.by_bucket.count[blockIdx.x + 1];
  for (unsigned w = threadIdx.x; w < n_local * 2; w += 512) reinterpret_cast<uint4*>(slots)[w] = make_uint4(~0u, ~0u, ~0u, ~0u);
  if (threadIdx.x == 0) n_over = 0;
  constexpr int kItems = 4;
  for (unsigned i0 = begin; i0 < end; i0 += 512 * kItems) {
    unsigned key[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const unsigned i = i0 + 512 * j + threadIdx.x;
      key[j] = i < end ? sc.keys[i] : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      if (i0 + 512 * j + threadIdx.x >= end) break;
      const unsigned m = hs_mix32(key[j]);
      if (m == B::kFree) { *const_cast<unsigned*>(hs_special(hs)) = 1u; continue; }
      bool done = false;
      for (unsigned b = __umulhi(m, (unsigned)hs.n_buckets) - b0; b < n_local && !done; ++b) {
        B k;
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(slots + b * B::kSlots);
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(k.w[0]), "=r"(k.w[1]), "=r"(k.w[2]), "=r"(k.w[3]) : "r"(at) : "memory");
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(k.w[4]), "=r"(k.w[5]), "=r"(k.w[6]), "=r"(k.w[7]) : "r"(at + 16) : "memory");
        done = k.has(m);
        for (int s = k.first_free(); s < B::kSlots && !done; ++s) {
          const unsigned cur = atomicCAS(slots + b * B::kSlots + s, B::kFree, m);
          done = cur == B::kFree || cur == m;
        }
      }
      if (!done) sc.keys[begin + atomicAdd(&n_over, 1u)] = key[j];
    }
  }
  bulk_fence();
  __syncthreads();
  if (threadIdx.x == 0) {
    bulk_store<false>(reinterpret_cast<uint4*>(hs.slots) + (size_t)b0 * 2, slots, n_local * kBucketBytes);
    sc.n_over[blockIdx.x] = n_over;
    bulk_wait();
  }
}
// (one warp per part)
__global__ void __launch_bounds__(256) part_over_kernel(HashSetView hs, BuildScratch sc, int* status) {
  const int part = (int)(blockIdx.x * 8 + (threadIdx.x >> 5));
  if (part >= sc.by_bucket.parts) return;
  const unsigned begin = sc.by_bucket.count[part], n = sc.n_over[part];
  for (unsigned i = threadIdx.x & 31; i < n; i += 32)
    if (hs_insert<true>(hs, sc.keys[begin + i]) < 0) atomicOr(status, kStHashFull);
}

// The shorter prefixes, all in direct regions.  A thread gathers one word of the bits behind a prefix of n = L - 2 codes
// (neighbouring threads: neighbouring prefixes, whose bits in sc.any are neighbours), and enters the prefix further up where it
// begins an item.
__global__ void __launch_bounds__(256) part_up_kernel(LevelInfo li, PrefixMapView pm, BuildScratch sc, int n, int* status) {
  const unsigned q_count = (unsigned)li.mult[n], q = blockIdx.x * 256 + threadIdx.x, t0 = blockIdx.y * 64;
  if (q >= q_count) return;
  const int nt = min(64, li.T[n] - (int)t0);
  unsigned long long word = 0;
#pragma unroll 16
  for (int t = 0; t < nt; ++t) {
    const unsigned p = q + (t0 + t) * q_count;
    word |= (unsigned long long)((sc.any[p >> 5] >> (p & 31)) & 1u) << t;
  }
  pm.slots[pm.level_off[n] + (unsigned long long)q * pm.set_words + blockIdx.y] = word;
  if (!word) return;
  unsigned p = q;
  int r = 1;
  for (int lv = n - 1; lv >= 0 && r > 0; --lv) {        // (as in set_build_kernel)
    const unsigned c = p / (unsigned)li.mult[lv];
    p -= c * (unsigned)li.mult[lv];
    r = pm_add(pm, lv, p, (int)c, false);
  }
  if (r < 0) atomicOr(status, kStHashFull);
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

// Fills in the sizes of a build by parts, or leaves on = 0 where it does not apply (wide keys, a hashed region, more than
// kBuildMaxParts parts) or does not pay: its eight launches and its passes over all counters cost some 40 us, so it starts at
// 1.5M items; a region of less than 16 MB has too few parts for the chip.  One pass -> by parts, us: 0.6M items 68 -> 92, 1M
// 81 -> 96 (8 MB) and 90 -> 103 (17 MB), 1.2M 104 -> 104 (34 MB), 2M 129 -> 117 (17 MB), 4M 228 -> 176 (34 MB) and 192 -> 179
// (8 MB), 12M 672 -> 366 (34 MB).
// (A part is at most 64 KB, so that three blocks of an SM overlap their phases.)
constexpr unsigned long long kBuildMinItems = 3ull << 19, kBuildMinRegion = 16ull << 20;
void plan_build(const LevelInfo& li, HashSetView hs, PrefixMapView pm, unsigned long long n, BuildScratch* sc) {
  *sc = BuildScratch{};
  if (li.L < 2 || !hs.narrow || n < kBuildMinItems || n >= 1ull << 31) return;
  for (int l = 0; l < li.L; ++l)
    if (pm.level_slots[l] != 0) return;                  // (a direct longest region means that the shorter ones are direct too)
  const unsigned long long prefixes = li.mult[li.L - 1];
  if (prefixes * pm.set_words * 8 < kBuildMinRegion) return;
  auto deal = [](unsigned long long things, int bytes_each, BuildDeal* dl) {
    while ((2ull << dl->shift) * bytes_each <= 64u << 10) ++dl->shift;
    const unsigned long long parts = (things + (1ull << dl->shift) - 1) >> dl->shift;
    dl->parts = (int)(parts <= kBuildMaxParts ? parts : 0);
    return dl->parts != 0;
  };
  sc->on = deal(prefixes, pm.set_words * 8, &sc->by_prefix) && deal(hs.n_buckets, kBucketBytes, &sc->by_bucket);
}

// Clears both tables and enters the n items; *n_unique = how many of them are distinct.
cudaError_t launch_set_build(const LevelInfo& li, HashSetView hs, PrefixMapView pm, const BuildScratch& sc, const int* codes,
                      unsigned long long n, unsigned long long* n_unique, int* status, int n_sm, cudaStream_t st) {
  const bool vec = codes_vec(li, codes);
  if (sc.on) {
    const int last = li.L - 1;
    const unsigned prefixes = (unsigned)li.mult[last], run = (unsigned)((n + kBuildBlocks - 1) / kBuildBlocks);
    const KeySplit split{prefixes, nextafterf((float)(1.0 / (double)prefixes), 0.f)};
    const DealPrefix by_prefix{split, sc.by_prefix.shift};
    const DealBucket by_bucket{(unsigned)hs.n_buckets, sc.by_bucket.shift};
    const int both = sc.by_prefix.parts + sc.by_bucket.parts;
    const int bits_bytes = (1 << sc.by_prefix.shift) * pm.set_words * 8 + (1 << sc.by_prefix.shift) / 8;
    const int slots_bytes = kBucketBytes << sc.by_bucket.shift;
    // the packed keys wait in the hash set's slots, which are at least as many as the items, until they have been dealt out twice
    unsigned* keys = reinterpret_cast<unsigned*>(hs.slots);
    cudaError_t failed = cudaSuccess;
    auto go = [&](auto kernel, dim3 grid, int threads, int bytes, auto... args) {
      if (failed != cudaSuccess) return;
      // (the limit that needs no attribute, 48 KB, counts the kernel's static shared memory too)
      if (bytes > 32 << 10) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      LaunchScope ls(kcHash, st);
      kernel<<<grid, threads, bytes, st>>>(args...);
      failed = cudaGetLastError();                   // (taken, so that the call after this one does not report it again)
    };
    auto deal = [&](auto kernel, const BuildDeal& dl, auto part_of) {
      go(kernel, kBuildBlocks, 1024, (kDealKeys + 2 * dl.parts) * 4, dl, part_of, (const unsigned*)sc.n_valid, (unsigned)n, run, (const unsigned*)keys, sc.keys);
    };
    // (the longest region is the last, and written whole)
    cudaMemsetAsync(sc.by_prefix.count, 0, (size_t)(both + 2) * sizeof(unsigned), st);
    static_assert(2 * kBuildMaxParts * 4 + 16 + kCountRingBytes <= (227 << 10) - 1024, "the ring beside both deals' counters");
    const bool ring = vec && li.L == 4;
    go(ring ? part_count_kernel<true, true> : vec ? part_count_kernel<true, false> : part_count_kernel<false, false>, kBuildBlocks, 1024,
       both * 4 + (ring ? 16 + kCountRingBytes : 0), li, hs, pm, sc, by_bucket, codes, (unsigned)n, run, keys, n_unique, status);
    go(part_scan_kernel, 2, 1024, 0, sc);
    deal(part_deal_kernel<DealPrefix>, sc.by_prefix, by_prefix);
    go(part_bits_kernel, sc.by_prefix.parts, 512, bits_bytes, pm, sc, last, split, n_unique);
    go(part_up_kernel, dim3((unsigned)((li.mult[last - 1] + 255) / 256), (li.T[last - 1] + 63) / 64), 256, 0, li, pm, sc, last - 1, status);
    deal(part_deal_kernel<DealBucket>, sc.by_bucket, by_bucket);
    go(part_slots_kernel, sc.by_bucket.parts, 512, slots_bytes, hs, sc);
    go(part_over_kernel, (sc.by_bucket.parts + 7) / 8, 256, 0, hs, sc, status);
    return failed;
  }
  cudaMemsetAsync(n_unique, 0, sizeof(unsigned long long), st);
  cudaMemsetAsync(hs.slots, 0xff, (size_t)hs.n_buckets * kBucketBytes, st);
  cudaMemsetAsync(hs.slots + hs.n_buckets * (kBucketBytes / 8), 0, kBucketBytes, st);      // the special word (HashSetView)
  cudaMemsetAsync(pm.slots, 0, (size_t)pm.n_words * sizeof(unsigned long long), st);
  if (!n) return cudaSuccess;
  LaunchScope ls(kcHash, st);
  const unsigned long long blocks = (n + 255) / 256;
  const unsigned grid = (unsigned)(blocks < 8ull * n_sm ? blocks : 8ull * n_sm);
  auto go = [&](auto kernel) { kernel<<<grid, 256, 0, st>>>(li, hs, pm, codes, n, n_unique, status); };
  if (vec) { if (hs.narrow) go(set_build_kernel<true, true>); else go(set_build_kernel<true, false>); }
  else { if (hs.narrow) go(set_build_kernel<false, true>); else go(set_build_kernel<false, false>); }
  return cudaGetLastError();
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
