// sr_cal.cuh -- device code shared by the CAL finder's kernels: seed lookups in
// the index forms (DevIndex), a read's packed codes and k-mers, block-wide sort
// and prefix sum.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "sr_internal.h"
#include "sr_seed.h"

namespace sr {
namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr uint64_t kCalBias = 1024;
constexpr uint64_t kCalMask = (1ull << 59) - 1;
constexpr uint64_t kNoKey = ~0ull;

__device__ __forceinline__ uint64_t cal_key(uint32_t ref, uint32_t strand, int64_t cal) {
  return (static_cast<uint64_t>(ref) << 60) | (static_cast<uint64_t>(strand) << 59) |
         static_cast<uint64_t>(cal + static_cast<int64_t>(kCalBias));
}

// ASCII -> 2-bit code; 4 for a non-ACGT byte
__device__ __forceinline__ uint32_t code_of(char ch) {
  switch (static_cast<unsigned>(static_cast<unsigned char>(ch)) | 0x20u) {
    case 'a': return 0;
    case 'c': return 1;
    case 'g': return 2;
    case 't': return 3;
    default: return 4;
  }
}

// the end of the run of keys equal to key that starts at l (l itself when K[l]
// differs): doubling steps, then a binary search, so that a repeat's run of
// thousands of entries costs tens of dependent loads and a run of one costs one
template <typename KT>
__device__ __forceinline__ uint64_t run_end(const KT* K, uint64_t l, uint64_t s1, uint32_t key) {
  if (l >= s1 || K[l] != key) return l;
  uint64_t in = l, step = 1;  // K[in] == key
  while (in + step < s1 && K[in + step] == key) {
    in += step;
    step <<= 1;
  }
  uint64_t out = in + step < s1 ? in + step : s1;  // s1, or K[out] != key
  while (in + 1 < out) {
    const uint64_t mid = in + ((out - in) >> 1);
    if (K[mid] == key) in = mid;
    else out = mid;
  }
  return out;
}

// entries [lo, hi) of the sorted keys K[s0 .. s1) equal to key
template <typename KT>
__device__ __forceinline__ void key_range(const KT* K, uint64_t s0, uint64_t s1, uint32_t key, uint64_t* lo,
                                          uint64_t* hi) {
  uint64_t l = s0, u = s1;
  while (l < u) {
    const uint64_t mid = l + ((u - l) >> 1);
    if (K[mid] < key) l = mid + 1;
    else u = mid;
  }
  *lo = l;
  *hi = run_end(K, l, s1, key);
}

// packed index: entries [lo, hi) of reference r with key `key` in bucket b
// (16-bit keys in key16, 32-bit ones in key)
__device__ __forceinline__ void lookup_packed(const DevIndex& di, uint64_t b, uint32_t key, int r, uint64_t* lo,
                                              uint64_t* hi) {
  const uint64_t s0 = di.jptr[b * di.n_refs + r], s1 = di.jptr[(b + 1) * di.n_refs + r];
  if (di.key_bits == 16) key_range(di.key16[r], s0, s1, key, lo, hi);
  else key_range(di.key[r], s0, s1, key, lo, hi);
}

// 32 aligned bytes, used once (no L1 line kept), as one request
__device__ __forceinline__ void ld_once_32(const uint32_t* p, uint32_t (&v)[8]) {
  asm("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "l"(p));
}

// bits 0 and 1: the low and the high half of w equal key (kk: it in both halves).
// A half of w ^ kk is zero exactly when adding 0x7fff to its low 15 bits leaves
// its top bit clear and its top bit was clear.
__device__ __forceinline__ uint32_t halves_equal(uint32_t w, uint32_t kk) {
  const uint32_t x = w ^ kk;
  const uint32_t z = ~(((x & 0x7fff7fffu) + 0x7fff7fffu) | x) & 0x80008000u;
  return ((z >> 15) & 1u) | (z >> 30);
}

// packed index with bucket heads: entries [lo0, hi0) of reference 0 and [lo1,
// hi1) of reference 1 with key `key` in bucket b, from the bucket's head alone
// (an empty range may start anywhere); false when the bucket spilled (its
// entries are then looked up in jptr and the keys).
//
// Random reads of a table past the L2 are bound by the number of 32-byte requests,
// each of which moves about 106 bytes of DRAM: 293 G/s over 32 MB, 76 over 256 MB,
// 59 over 512 MB and 54 over 1 GB (6.3 TB/s of DRAM), and 64 bytes as two of them
// at half that.  So the counts and the first keys lie in the first 32 bytes, and
// the others are read only where a bucket has more: 300k xenograft reads against
// 2 x 16 Mbp 1.21 ms with one 64-byte head per seed, 0.77 with 32.
__device__ __forceinline__ bool lookup_head(const DevIndex& di, uint64_t b, uint32_t key, uint32_t* lo0, uint32_t* hi0,
                                            uint32_t* lo1, uint32_t* hi1) {
  const uint32_t* h = di.heads + b * static_cast<uint32_t>(di.head_words);
  uint32_t v[8];
  ld_once_32(h, v);
  if (v[2] == kHeadSpill) return false;
  const uint32_t n0 = v[2] & 0xffu, n1 = (v[2] >> 8) & 0xffu;
  uint32_t eq = 0;  // bit i: key i of the head
  if (di.key_bits == 16) {
    const uint32_t kk = key | (key << 16);
#pragma unroll
    for (int j = 0; j < 6; ++j) eq |= halves_equal(v[2 + j], kk) << (2 * j);
    eq >>= 1;  // the first half holds the counts
    if (n0 + n1 > static_cast<uint32_t>(kHeadNear16)) {
      uint32_t u[8];
      ld_once_32(h + 8, u);
#pragma unroll
      for (int j = 0; j < 8; ++j) eq |= halves_equal(u[j], kk) << (kHeadNear16 + 2 * j);
    }
  } else {
#pragma unroll
    for (int j = 0; j < kHeadNear32; ++j) eq |= (v[3 + j] == key ? 1u : 0u) << j;
    if (n0 + n1 > static_cast<uint32_t>(kHeadNear32)) {
      uint32_t u[8];
      ld_once_32(h + 8, u);
#pragma unroll
      for (int j = 0; j < 8; ++j) eq |= (u[j] == key ? 1u : 0u) << (kHeadNear32 + j);
    }
  }
  // equal keys are consecutive within each reference's run of sorted keys
  const uint32_t m0 = (1u << n0) - 1u, m1 = ((1u << (n0 + n1)) - 1u) & ~m0;
  const uint32_t e0 = eq & m0, e1 = eq & m1;
  *lo0 = v[0] + (e0 ? __ffs(e0) - 1u : 0u);
  *hi0 = *lo0 + __popc(e0);
  *lo1 = v[1] + (e1 ? __ffs(e1) - 1u - n0 : 0u);
  *hi1 = *lo1 + __popc(e1);
  return true;
}

// entries [lo, hi) of reference r whose key equals the seed's
__device__ __forceinline__ void lookup(const DevIndex& di, int r, uint64_t canon, uint64_t* lo, uint64_t* hi) {
  const int kb = 2 * (di.k - di.a);
  const uint64_t h = seed_hash(canon, di.k, di.hash_seed[r]);
  const uint64_t b = h >> kb;
  const uint32_t key = static_cast<uint32_t>(h & mask_bits(kb));
  uint64_t s0 = di.ptr[r][b], s1 = di.ptr[r][b + 1];
  const uint32_t* K = di.key[r];
  // lower bound of key in the bucket
  uint64_t l = s0, u = s1;
  while (l < u) {
    const uint64_t mid = l + ((u - l) >> 1);
    if (K[mid] < key) l = mid + 1;
    else u = mid;
  }
  *lo = l;
  *hi = run_end(K, l, s1, key);
}

// read r's codes into shared memory; false (and status) on a non-ACGT base
__device__ __forceinline__ bool load_codes(const char* bases, uint64_t o0, uint32_t m, uint8_t* q, int lane,
                                           uint32_t* status) {
  bool bad = false;
  for (uint32_t t = lane; t < m; t += 32) {
    const uint32_t c = code_of(bases[o0 + t]);
    bad |= c > 3;
    q[t] = static_cast<uint8_t>(c & 3);
  }
  bad = __any_sync(FULL, bad);
  if (bad && lane == 0) atomicOr(status, kStBadBase);
  __syncwarp();
  return !bad;
}

// The read's codes as 2-bit fields, first base highest, in kPackWords 32-bit
// words (kMaxReadLen bases and two words of padding): Pk for the read, Rk for
// the reverse complement of the read padded to kMaxReadLen bases, so that a
// seed's forward and reverse-complement k-mers (Kmer's fwd and rc) are each
// read with two funnel shifts.  Bases past the read's end are never extracted.
constexpr int kPackWords = kMaxReadLen / 16 + 2;

// q: the codes (one byte each, 4-byte aligned); lanes 0-15 pack word j
__device__ __forceinline__ void pack_codes(const uint8_t* q, uint32_t* Pk, uint32_t* Rk, int lane) {
  const uint32_t* q32 = reinterpret_cast<const uint32_t*>(q);
  uint32_t w = 0;
  if (lane < kMaxReadLen / 16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // four codes, first in byte 0, to one byte with the first code highest
      const uint32_t x = __byte_perm(q32[4 * lane + i] & 0x03030303u, 0, 0x0123);
      const uint32_t t = (x | (x >> 6)) & 0x000F000Fu;
      w = (w << 8) | ((t | (t >> 12)) & 0xFFu);
    }
  }
  // the reverse complement: words in reverse order, 2-bit fields reversed, complemented
  const uint32_t src = __shfl_sync(FULL, w, (kMaxReadLen / 16 - 1 - lane) & 31);
  uint32_t r = __brev(~src);
  r = ((r >> 1) & 0x55555555u) | ((r << 1) & 0xAAAAAAAAu);
  if (lane < kMaxReadLen / 16) {
    Pk[lane] = w;
    Rk[lane] = r;
  } else if (lane < kPackWords) {
    Pk[lane] = 0;
    Rk[lane] = 0;
  }
  __syncwarp();
}

// the k bases at o of a packed string, first base highest (k <= 32)
__device__ __forceinline__ uint64_t kmer_at(const uint32_t* W, uint32_t o, int k) {
  const uint32_t b = 2 * o, j = b >> 5, s = b & 31;
  const uint32_t w0 = W[j], w1 = W[j + 1], w2 = W[j + 2];
  const uint64_t win = (static_cast<uint64_t>(__funnelshift_l(w1, w0, s)) << 32) | __funnelshift_l(w2, w1, s);
  return win >> (64 - 2 * k);
}

// a kept lookup: first matching entry (38 bits), their number (24 bits) and the
// seed's orientation bits (2)
constexpr uint32_t kRangeCntMax = (1u << 24) - 1u;
constexpr uint64_t kRangeLoMax = (1ull << 38) - 1ull;
__device__ __forceinline__ uint64_t range_pack(uint64_t lo, uint32_t cnt, uint32_t rori) {
  return (lo << 26) | (static_cast<uint64_t>(cnt) << 2) | rori;
}

// block-wide bitonic sort of P (a power of two) keys, ascending
__device__ void bitonic(uint64_t* s, uint32_t P) {
  for (uint32_t size = 2; size <= P; size <<= 1) {
    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
      for (uint32_t i = threadIdx.x; i < P / 2; i += blockDim.x) {
        const uint32_t lo = 2 * i - (i & (stride - 1));
        const uint32_t hi = lo + stride;
        const bool up = (lo & size) == 0;
        const uint64_t x = s[lo], y = s[hi];
        if ((x > y) == up) {
          s[lo] = y;
          s[hi] = x;
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ uint32_t pow2_at_least(uint32_t n) {
  uint32_t p = 1;
  while (p < n) p <<= 1;
  return p;
}

// Block-wide exclusive prefix sum of one 64-bit value per thread; *total gets
// the block's sum.  (Two 32-bit counts packed as high:low add without carries
// while each total stays below 2^32.)
__device__ uint64_t block_exscan(uint64_t v, uint64_t* total) {
  __shared__ uint64_t warp_sum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(FULL, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sum[w] = x;
  __syncthreads();
  if (w == 0) {
    uint64_t t = lane < nw ? warp_sum[lane] : 0ull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(FULL, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) warp_sum[lane] = t;
  }
  __syncthreads();
  const uint64_t before = (w ? warp_sum[w - 1] : 0ull) + x - v;
  *total = warp_sum[nw - 1];
  __syncthreads();
  return before;
}

}  // namespace
}  // namespace sr
