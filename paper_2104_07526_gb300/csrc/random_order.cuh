// Random orders: records (or batches) sorted by the high 32 bits of a
// SplitMix64 output per input index, ties by index.  Included by reorder.cu.
//
// The keys are as good as uniform, so the sort goes from the top: one or two
// partition passes split the sequence into buckets, equal ranges of keys of
// kBucketMean elements on average, and a last pass sorts each bucket in
// shared memory and writes it out.  What a partition pass leaves inside a
// bucket is in no particular order: each element carries its index, the last
// pass sorts by (key, index), and the result is the same whatever order the
// elements arrived in.  So a pass needs no stable ranks (one shared-memory
// atomic per element instead of a warp-wide match) and no counts per tile (a
// tile reserves its part of each bucket with one atomic add on the bucket's
// cursor), and keys are never stored: each pass computes them from the index.
//   1. k_random_count (first pass: from the index alone; second: from the
//      indices it will move) counts the buckets; a scan of the counts gives
//      every bucket its first position: the cursors.
//   2. k_random_partition moves records and indices; the cursors end at the
//      buckets' ends.
//   3. k_random_finish sorts the buckets.
// A bucket larger than its block's shared memory (which uniform keys do not
// give, but a seed cannot be shown never to give) is sorted by counting, one
// comparison per pair of its elements.
//
// Per record the passes move 16 + 20, 4 + 20 + 20 and 20 + 16 bytes (with a
// permutation output 4 more): 116, against 172 for four stable 8-bit passes
// that carry key and record, which this replaced.  Bounds and times at 50M
// records (ncu): the partition passes, 0.34 and 0.35 ms, are bound by their
// shared-memory steps between barriers at 66-69% of the DRAM throughput; the
// finish, 0.51 ms, by instruction issue (60% of slots) of the key arithmetic
// and the comparisons inside bins.  50M with permutation 2.60 -> 1.35 ms.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace pcr {
namespace {

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014): output k of the generator
// seeded with `seed` mixes the state seed + (k + 1) * 0x9E3779B97F4A7C15.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t k) {
  uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Sort key of input index i.
__device__ __forceinline__ uint32_t random_key(uint64_t seed, uint32_t i) {
  return static_cast<uint32_t>(splitmix64(seed, i) >> 32);
}

// Partition tiles of 4096 elements (2 blocks of 512 threads per SM): longer
// runs per digit than tiles of 2048 (50M records with both passes 1.78
// against 2.02 ms).
constexpr int kPartThreads = 512;
constexpr int kPartRounds = 8;  // elements per thread
constexpr uint32_t kPartTile = kPartThreads * kPartRounds;
constexpr int kMaxPassBits = 11;
// Up to this many buckets, one pass splits them all (2.1M records with
// their permutation: 97 us, in two passes 128).
// Debug builds split batch orders (no records) in two passes from 9 buckets on,
// 2.03M points, where release builds take 520M.
#ifdef PCR_DEBUG
template <bool REC>
constexpr uint32_t kOnePassBuckets = REC ? 1u << kMaxPassBits : 8u;
#else
template <bool REC>
constexpr uint32_t kOnePassBuckets = 1u << kMaxPassBits;
#endif
// Buckets of about 2000 elements, four blocks of 256 threads per SM; twice
// that with 512 threads measured within 2% (50M: 1.59 and 1.63 ms, 400M:
// 13.9 and 13.8).
constexpr int kFinishThreads = 256;
constexpr int kFinishRounds = 9;
constexpr uint32_t kFinishCap = kFinishThreads * kFinishRounds;
// Elements a bucket has on average, at most: 7 standard deviations below the
// capacity.
constexpr uint32_t kBucketMean = 1984;
constexpr int kBinBits = 12;  // 8192 bins: 1.87 against 1.78 ms at 50M
constexpr uint32_t kBins = 1u << kBinBits;
constexpr uint32_t kPosBits = 13;  // a bucket position in a packed word
static_assert(kPartTile <= 1u << 12, "a tile slot and a digit share one word");
static_assert(kFinishCap <= 1u << kPosBits, "a position and the key's leading bits share one word");
static_assert(kBins % (2 * kFinishThreads) == 0, "whole words of two bins per thread");

// A sequence is split into `buckets` equal ranges of keys.  With two passes
// the first one goes by bucket >> `second`, the second by the low bits.
struct RandomSplit {
  int passes;
  uint32_t buckets;
  int second;
};

template <bool REC>
constexpr RandomSplit random_split(uint32_t count) {
  const uint32_t buckets = count / kBucketMean + (count % kBucketMean != 0);
  if (buckets <= 1) return {0, 1u, 0};
  if (buckets <= kOnePassBuckets<REC>) return {1, buckets, 0};
  int bits = 0;
  while ((buckets - 1) >> bits) ++bits;
  return {2, buckets, bits / 2};
}

// Digits of each pass.
constexpr uint32_t first_digits(RandomSplit p) { return ((p.buckets - 1) >> p.second) + 1; }
constexpr uint32_t second_digits(RandomSplit p) { return 1u << p.second; }
static_assert(first_digits(random_split<true>(0xFFFFFFFFu)) <= 1u << kMaxPassBits &&
                  second_digits(random_split<true>(0xFFFFFFFFu)) <= 1u << kMaxPassBits,
              "both digits of the largest split fit a pass");

// First counter of the second pass (a multiple of four words), and the words
// of counters a split needs.
constexpr uint64_t second_counters(RandomSplit p) { return (first_digits(p) + 3u) & ~3u; }
template <bool REC>
constexpr uint64_t random_counter_words(uint32_t count) {
  const RandomSplit p = random_split<REC>(count);
  return p.passes == 0 ? 0 : second_counters(p) + (p.passes == 2 ? p.buckets : 0);
}

// Bucket of a key, and its place inside the bucket's range: both grow with
// the key, and keys of one bucket differ exactly when their places do.
__device__ __forceinline__ uint32_t bucket_of(uint32_t key, uint32_t buckets) { return __umulhi(key, buckets); }
__device__ __forceinline__ uint32_t place_of(uint32_t key, uint32_t buckets) { return key * buckets; }

__global__ void __launch_bounds__(256) k_zero_words(uint32_t* __restrict__ p, uint64_t count) {
  after_previous();
  for (uint64_t i = blockIdx.x * 256ull + threadIdx.x; i < count; i += gridDim.x * 256ull) p[i] = 0u;
}

// First pass: elements per top digit, from the indices 0 .. count - 1.
__global__ void __launch_bounds__(kPartThreads) k_random_count_first(uint32_t count, uint64_t seed, uint32_t buckets,
                                                                     int second, uint32_t radix,
                                                                     uint32_t* __restrict__ counts) {
  after_previous();
  extern __shared__ __align__(16) uint32_t s_count[];
  for (uint32_t d = threadIdx.x; d < radix; d += kPartThreads) s_count[d] = 0u;
  __syncthreads();
  for (uint64_t i = blockIdx.x * static_cast<uint64_t>(kPartThreads) + threadIdx.x; i < count;
       i += gridDim.x * static_cast<uint64_t>(kPartThreads))
    atomicAdd(&s_count[bucket_of(random_key(seed, static_cast<uint32_t>(i)), buckets) >> second], 1u);
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < radix; d += kPartThreads)
    if (s_count[d]) atomicAdd(counts + d, s_count[d]);
}

// Second pass: elements per bucket of the whole split, from the indices the
// first pass left (in runs of equal first digit, so a chunk holds one or a
// few first digits).
constexpr uint32_t kCountChunk = 16384;
__global__ void __launch_bounds__(kPartThreads) k_random_count_second(const uint32_t* __restrict__ iin, uint32_t count,
                                                                      uint64_t seed, uint32_t buckets, int second,
                                                                      uint32_t* __restrict__ counts) {
  after_previous();
  extern __shared__ __align__(16) uint32_t s_count[];
  const uint32_t radix = 1u << second;
  const uint64_t first = blockIdx.x * static_cast<uint64_t>(kCountChunk);
  const uint64_t end = first + kCountChunk < count ? first + kCountChunk : count;
  const uint32_t lo = bucket_of(random_key(seed, iin[first]), buckets) >> second;
  const uint32_t hi = bucket_of(random_key(seed, iin[end - 1]), buckets) >> second;
  for (uint32_t part = lo; part <= hi; ++part) {
    for (uint32_t d = threadIdx.x; d < radix; d += kPartThreads) s_count[d] = 0u;
    __syncthreads();
    for (uint64_t i = first + threadIdx.x; i < end; i += kPartThreads) {
      const uint32_t b = bucket_of(random_key(seed, __ldg(iin + i)), buckets);
      if ((b >> second) == part) atomicAdd(&s_count[b & (radix - 1)], 1u);
    }
    __syncthreads();
    for (uint32_t d = threadIdx.x; d < radix; d += kPartThreads)
      if (s_count[d]) atomicAdd(counts + ((part << second) | d), s_count[d]);
    __syncthreads();
  }
}

template <bool REC>
constexpr size_t partition_smem(uint32_t radix) {
  return (REC ? sizeof(uint4) * kPartTile : 0) + 2 * sizeof(uint32_t) * kPartTile +
         2 * sizeof(uint32_t) * radix;
}

// One partition pass over a tile of kPartTile elements.  The records come in
// with asynchronous copies while the elements find their digits; a shared
// atomic per element gives its place among the tile's elements of its digit, a
// scan of the counts the tile's digit order, and one atomic add per digit on
// its bucket's cursor the place of the tile's run in the bucket.  The tile then
// leaves in digit order, so each digit's run is one contiguous store.  FIRST:
// element i's index is i; else iin[i], and the elements of a tile may belong
// to several buckets of the first pass, which are moved one after the other.
template <bool REC, bool FIRST>
__global__ void __launch_bounds__(kPartThreads, 2)
    k_random_partition(const uint4* __restrict__ rin, const uint32_t* __restrict__ iin, uint4* __restrict__ rout,
                       uint32_t* __restrict__ iout, uint32_t n, uint64_t seed, uint32_t buckets, int second,
                       uint32_t radix, uint32_t* __restrict__ cursors) {
  after_previous();
  extern __shared__ __align__(16) unsigned char s_bytes[];
  uint4* s_rec = reinterpret_cast<uint4*>(s_bytes);                                      // [kPartTile] with REC
  uint32_t* s_idx = reinterpret_cast<uint32_t*>(s_bytes + (REC ? sizeof(uint4) * kPartTile : 0));  // [kPartTile]
  uint32_t* s_ord = s_idx + kPartTile;                                                   // [kPartTile]
  uint32_t* s_base = s_ord + kPartTile;                                                  // [radix]
  uint32_t* s_delta = s_base + radix;                                                    // [radix]
  __shared__ uint32_t s_part[2];
  const uint32_t t = threadIdx.x;
  const uint64_t tile_base = static_cast<uint64_t>(blockIdx.x) * kPartTile;
  const uint32_t valid = static_cast<uint32_t>(n - tile_base < kPartTile ? n - tile_base : kPartTile);
  // the indices before the records: they would otherwise wait behind the
  // tile's 64 KB
  uint32_t b[kPartRounds];  // the element's index, then its first digit (FIRST) or bucket
#pragma unroll
  for (int r = 0; r < kPartRounds; ++r) {
    const uint32_t j = r * kPartThreads + t;
    b[r] = FIRST ? static_cast<uint32_t>(tile_base) + j : j < valid ? __ldg(iin + tile_base + j) : 0u;
  }
  if constexpr (REC) {
    for (uint32_t j = t; j < valid; j += kPartThreads) copy16_async(s_rec + j, rin + tile_base + j, 16u);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
#pragma unroll
  for (int r = 0; r < kPartRounds; ++r) {
    const uint32_t j = r * kPartThreads + t;
    if (j < valid) s_idx[j] = b[r];
    b[r] = bucket_of(random_key(seed, b[r]), buckets) >> (FIRST ? second : 0);
    if (!FIRST && j == 0) s_part[0] = b[r] >> second;
    if (!FIRST && j == valid - 1) s_part[1] = b[r] >> second;
  }
  uint32_t lo = 0, hi = 0;
  if constexpr (!FIRST) {
    __syncthreads();
    lo = s_part[0];
    hi = s_part[1];
  }
  for (uint32_t part = lo; part <= hi; ++part) {
    for (uint32_t d = t; d < radix; d += kPartThreads) s_base[d] = 0u;
    __syncthreads();
    uint32_t rank[kPartRounds];
    auto mine = [&](int r) { return r * kPartThreads + t < valid && (FIRST || (b[r] >> second) == part); };
    auto digit = [&](int r) { return FIRST ? b[r] : b[r] & (radix - 1); };
#pragma unroll
    for (int r = 0; r < kPartRounds; ++r)
      rank[r] = mine(r) ? atomicAdd(&s_base[digit(r)], 1u) : 0u;
    __syncthreads();
    // exclusive scan of the counts; thread t owns `per` consecutive digits
    const uint32_t per = (radix + kPartThreads - 1) / kPartThreads;
    const uint32_t d0 = t * per;
    uint32_t sum = 0;
    for (uint32_t k = 0; k < per; ++k) sum += d0 + k < radix ? s_base[d0 + k] : 0u;
    uint32_t total;
    uint32_t at = block_exclusive_scan<kPartThreads>(sum, total);
    for (uint32_t k = 0; k < per && d0 + k < radix; ++k) {
      const uint32_t c = s_base[d0 + k];
      s_base[d0 + k] = at;
      if (c) s_delta[d0 + k] = atomicAdd(cursors + ((part << second) + d0 + k), c) - at;  // modulo 2^32
      at += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kPartRounds; ++r) {
      if (!mine(r)) continue;
      const uint32_t d = digit(r);
      const uint32_t slot = s_base[d] + rank[r];
      if (debug_in_range(slot, kPartTile)) s_ord[slot] = (d << 12) | (r * kPartThreads + t);
    }
    if constexpr (REC) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll 4
    for (uint32_t l = t; l < total; l += kPartThreads) {
      const uint32_t o = s_ord[l];
      const uint32_t j = o & (kPartTile - 1);
      const uint32_t g = s_delta[o >> 12] + l;
      if (!debug_in_range(g, n)) continue;
      if constexpr (REC) rout[g] = s_rec[j];
      iout[g] = s_idx[j];
    }
    __syncthreads();  // the next part reuses the order
  }
}

// Shared memory of k_random_finish: a bucket's records and packed words, and
// the bins (two 16-bit counters a word).
template <bool REC>
constexpr size_t finish_smem() {
  return (REC ? sizeof(uint4) * kFinishCap : 0) + sizeof(uint32_t) * kFinishCap + sizeof(uint16_t) * (kBins + 2);
}

// Where k_random_finish puts an element of final position g and input index i:
// its record to dst[g] (with REC), i to perm[g], g to rank[i]; perm and rank
// may be null.
struct RandomOut {
  uint4* dst = nullptr;
  uint32_t* perm = nullptr;
  uint32_t* rank = nullptr;
};

// Sort bucket blockIdx.x of `buckets` (its end is ends[bucket]; one bucket is
// the whole sequence, its indices the positions) by (key, index).  The places
// of the keys in the bucket's range fall into kBins bins, half an element
// each: a shared atomic counts an element into its bin, a scan places the
// bins, and each element is compared with the others of its bin (by the
// place's leading bits; elements equal in those, a few per bucket, look each
// other up).  The records wait in shared memory, so `rin` may be out.dst;
// `spare` holds as many records as rin and is written only for a bucket too
// large for shared memory.
template <bool REC>
__global__ void __launch_bounds__(kFinishThreads, 4)
    k_random_finish(const uint4* rin, const uint32_t* __restrict__ iin, uint32_t n, uint64_t seed, uint32_t buckets,
                    const uint32_t* __restrict__ ends, RandomOut out, uint4* spare) {
  after_previous();
  extern __shared__ __align__(16) unsigned char s_bytes[];
  uint4* s_rec = reinterpret_cast<uint4*>(s_bytes);
  uint32_t* s_word = reinterpret_cast<uint32_t*>(s_bytes + (REC ? sizeof(uint4) * kFinishCap : 0));
  uint16_t* s_bin = reinterpret_cast<uint16_t*>(s_word + kFinishCap);  // [kBins + 1]
  uint32_t* s_two = reinterpret_cast<uint32_t*>(s_bin);                // the bins, two a word
  const uint32_t t = threadIdx.x;
  const uint32_t start = blockIdx.x ? __ldg(ends + blockIdx.x - 1) : 0u;
  const uint32_t end = buckets > 1u ? __ldg(ends + blockIdx.x) : n;
  const uint32_t m = end - start;
  if (m == 0u) return;
  auto index_of = [&](uint32_t j) { return iin ? __ldg(iin + start + j) : start + j; };
  auto place_of_index = [&](uint32_t i) { return place_of(random_key(seed, i), buckets); };
  auto put = [&](uint32_t g, uint32_t i) {
    if (out.perm) out.perm[g] = i;
    if (out.rank && debug_in_range(i, n)) out.rank[i] = g;
  };
  bool large = m > kFinishCap;
#ifdef PCR_DEBUG
  large = large || (blockIdx.x & 1u);  // debug builds send every other bucket this way
#endif
  if (large) {
    // each element's position is the number of elements before it in order
    for (uint32_t e0 = 0; e0 < m; e0 += kFinishThreads) {
      const uint32_t e = e0 + t;
      const uint32_t i = e < m ? index_of(e) : 0u;
      const uint32_t mine = place_of_index(i);
      uint32_t before = 0;
      for (uint32_t c = 0; c < m; c += kFinishCap) {
        const uint32_t len = m - c < kFinishCap ? m - c : kFinishCap;
        __syncthreads();
        for (uint32_t f = t; f < len; f += kFinishThreads) s_word[f] = place_of_index(index_of(c + f));
        __syncthreads();
        for (uint32_t f = 0; f < len; ++f)
          before += s_word[f] < mine || (s_word[f] == mine && index_of(c + f) < i);
      }
      if (e < m) {
        put(start + before, i);
        if constexpr (REC) (rin == out.dst ? spare : out.dst)[start + before] = rin[start + e];
      }
    }
    if constexpr (REC) {
      if (rin == out.dst) {
        __syncthreads();  // the block's own stores to `spare` are visible to it
        for (uint32_t e = t; e < m; e += kFinishThreads) out.dst[start + e] = spare[start + e];
      }
    }
    return;
  }
  // rounds past the bucket's end are skipped by the whole block
  auto rounds = [&](auto f) {
#pragma unroll
    for (int r = 0; r < kFinishRounds; ++r)
      if (static_cast<uint32_t>(r) * kFinishThreads < m) f(r, r * kFinishThreads + t, r * kFinishThreads + t < m);
  };
  uint32_t idx[kFinishRounds], word[kFinishRounds], at[kFinishRounds];
  rounds([&](int r, uint32_t j, bool in) { idx[r] = in ? index_of(j) : 0u; });
  if constexpr (REC) {
    for (uint32_t j = t; j < m; j += kFinishThreads) copy16_async(s_rec + j, rin + start + j, 16u);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (uint32_t k = t; k < kBins / 2; k += kFinishThreads) s_two[k] = 0u;
  __syncthreads();
  // the place's leading bits with the position below them; its leading
  // kBinBits bits are the bin
  rounds([&](int r, uint32_t j, bool in) {
    word[r] = (place_of_index(idx[r]) & ~((1u << kPosBits) - 1u)) | j;
    const uint32_t bin = word[r] >> (32 - kBinBits), high = 16u * (bin & 1u);
    at[r] = in ? (atomicAdd(&s_two[bin >> 1], 1u << high) >> high) & 0xFFFFu : 0u;
  });
  __syncthreads();
  constexpr int kOwn = kBins / 2 / kFinishThreads;  // words per thread
  uint32_t own[kOwn], sum = 0;
  static_assert(kOwn % 4 == 0, "a thread's words move as 16-byte vectors");
  uint4* mine4 = reinterpret_cast<uint4*>(s_two) + t * (kOwn / 4);
#pragma unroll
  for (int k = 0; k < kOwn; k += 4) {
    const uint4 v = mine4[k / 4];
    own[k] = v.x, own[k + 1] = v.y, own[k + 2] = v.z, own[k + 3] = v.w;
  }
#pragma unroll
  for (int k = 0; k < kOwn; ++k) sum += (own[k] & 0xFFFFu) + (own[k] >> 16);
  uint32_t total;
  uint32_t run = block_exclusive_scan<kFinishThreads>(sum, total);
#pragma unroll
  for (int k = 0; k < kOwn; ++k) {
    const uint32_t low = own[k] & 0xFFFFu;
    const uint32_t both = run | ((run + low) << 16);
    run += low + (own[k] >> 16);
    own[k] = both;
  }
#pragma unroll
  for (int k = 0; k < kOwn; k += 4) mine4[k / 4] = make_uint4(own[k], own[k + 1], own[k + 2], own[k + 3]);
  if (t == 0) s_bin[kBins] = static_cast<uint16_t>(total);
  __syncthreads();
  rounds([&](int r, uint32_t, bool in) {
    if (in) s_word[s_bin[word[r] >> (32 - kBinBits)] + at[r]] = word[r];
  });
  __syncthreads();
  rounds([&](int r, uint32_t, bool in) {
    if (!in) return;
    const uint32_t bin = word[r] >> (32 - kBinBits);
    const uint32_t first = s_bin[bin], last = s_bin[bin + 1];
    at[r] = first;
    if (last - first == 1u) return;
    for (uint32_t f = first; f < last; ++f) {
      const uint32_t other = s_word[f];
      bool before = other < word[r];
      if (((other ^ word[r]) >> kPosBits) == 0u && other != word[r]) {
        const uint32_t i = index_of(other & ((1u << kPosBits) - 1u));
        const uint32_t p = place_of_index(i), q = place_of_index(idx[r]);
        before = p < q || (p == q && i < idx[r]);
      }
      at[r] += before;
    }
  });
  __syncthreads();
  if (out.rank) {
    rounds([&](int r, uint32_t, bool in) {
      if (in && debug_in_range(idx[r], n)) out.rank[idx[r]] = start + at[r];
    });
  }
  // records, then indices, leave in final order through the words' array
  if constexpr (REC) {
    rounds([&](int r, uint32_t j, bool in) {
      if (in && debug_in_range(at[r], m)) s_word[at[r]] = j;
    });
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
#pragma unroll 3
    for (uint32_t j = t; j < m; j += kFinishThreads) __stcs(out.dst + start + j, s_rec[s_word[j]]);
  }
  if (out.perm) {
    __syncthreads();
    rounds([&](int r, uint32_t, bool in) {
      if (in && debug_in_range(at[r], m)) s_word[at[r]] = idx[r];
    });
    __syncthreads();
#pragma unroll 3
    for (uint32_t j = t; j < m; j += kFinishThreads) out.perm[start + j] = s_word[j];
  }
}

// Random order of n records in `pts` (REC; `copy` holds as many), or of n
// indices: see RandomOut.  idx: two buffers of n words; counters:
// random_counter_words<REC>(n) words, 16-byte aligned; partials: as exclusive_scan.
template <bool REC>
cudaError_t random_order(uint4* pts, uint4* copy, uint32_t n, uint64_t seed, uint32_t* const idx[2],
                         uint32_t* counters, uint32_t* partials, RandomOut out, cudaStream_t s, const Device& d) {
  const RandomSplit p = random_split<REC>(n);
  LaunchChain run{s};
  // The limit belongs to the kernel, for every stream and host thread: always
  // the most any size asks for.  A limit per call (98 to 115 KB by the digits)
  // could be lowered by another thread's call before this one's launch, which
  // then fails.  How many blocks an SM holds follows from what a launch asks for.
  auto allow = [&](auto kernel, size_t bytes) {
    if (run.error == cudaSuccess)
      run.error = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  };
  const uint4* rin = pts;
  const uint32_t* iin = nullptr;
  uint32_t* ends = nullptr;
  if (p.passes > 0) {
    const uint64_t words = random_counter_words<REC>(n);
    const uint32_t tiles = static_cast<uint32_t>((static_cast<uint64_t>(n) + kPartTile - 1) / kPartTile);
    const uint32_t radix = first_digits(p);
    uint32_t* first = counters;
    run(k_zero_words, static_cast<unsigned>(words / 256 + 1 < 256 ? words / 256 + 1 : 256), 256, 0, counters, words);
    const uint32_t blocks = tiles < 4u * d.num_sms ? tiles : 4u * d.num_sms;
    run(k_random_count_first, blocks, kPartThreads, sizeof(uint32_t) * radix, n, seed, p.buckets, p.second, radix,
                                                                               first);
    run(k_scan_partials, 1, 1024, 0, first, radix);
    allow(k_random_partition<REC, true>, partition_smem<REC>(1u << kMaxPassBits));
    run(k_random_partition<REC, true>, tiles, kPartThreads, partition_smem<REC>(radix), pts, nullptr, copy, idx[0], n, seed, p.buckets, p.second, radix, first);
    rin = copy;
    iin = idx[0];
    ends = first;
    if (p.passes == 2) {
      uint32_t* both = counters + second_counters(p);
      const uint32_t low = second_digits(p);
      const uint32_t chunks = static_cast<uint32_t>((static_cast<uint64_t>(n) + kCountChunk - 1) / kCountChunk);
      run(k_random_count_second, chunks, kPartThreads, sizeof(uint32_t) * low, idx[0], n, seed, p.buckets, p.second,
                                                                                both);
      if (run.error == cudaSuccess) run.error = exclusive_scan(both, p.buckets, partials, s);
      allow(k_random_partition<REC, false>, partition_smem<REC>(1u << kMaxPassBits));
      run(k_random_partition<REC, false>, tiles, kPartThreads, partition_smem<REC>(low), copy, idx[0], pts, idx[1], n, seed, p.buckets, p.second, low, both);
      rin = pts;
      iin = idx[1];
      ends = both;
    }
  }
  out.dst = pts;
  allow(k_random_finish<REC>, finish_smem<REC>());
  run(k_random_finish<REC>, p.buckets, kFinishThreads, finish_smem<REC>(), rin, iin, n, seed, p.buckets, ends, out,
                                                                              copy);
  return run.error;
}

}  // namespace
}  // namespace pcr
