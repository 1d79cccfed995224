// sr_find.cu -- the CAL finder and filter in one pass per read (McVicar et al.,
// arXiv 1805.00106, Sec. 3.2 CAL finder, Sec. 3.3 CAL filter): seed lookups,
// equal CALs counted as they are found, the distinct ones sorted and merged into
// windows.  Same windows, in the same order, as the host stage sr_candidates.
//
// A true location gives the same CAL from most of a read's seeds, so a read has
// far fewer distinct CALs than CALs (a 100-base xenograft read: 68 CALs, about
// 4 runs of equal ones; a read in a tandem repeat of 100 copies: 20,000 CALs,
// about 110 distinct).  Only distinct CALs with their counts are sorted, and no
// lookup, CAL or window count goes through device memory between passes.
//
//   k_find_warp   one warp per read.  The entries of a round's 32 seeds are
//                 taken rank by rank (every seed's first entry, then every
//                 seed's second, ...): entries of one key are sorted by position,
//                 so one rank mostly holds one copy's CAL 32 times, which a
//                 ballot folds into one (CAL, count) run.  Up to kRuns runs and
//                 kRanks ranks; other reads are listed for
//   k_find_block  one block per read, the CALs counted in a hash table in shared
//                 memory (768, then 12288 distinct ones); reads with more are
//                 listed for the large-read path (sr_cal.cu).
//   k_find_out    the windows, staged in any order, into the list's arrays.
#include <cuda_runtime.h>
#include <stdint.h>

#include "sr_cal.cuh"
#include "sr_internal.h"

namespace sr {
namespace {

// a CAL as one key: ref (4 bits) | strand (1) | cal + 1024 (33), sorted as (ref,
// strand, cal); an element is the key above kCntBits bits of its count
constexpr int kCalBits = 33;
constexpr int kCntBits = 26;
constexpr uint32_t kCntMask = (1u << kCntBits) - 1u;
constexpr uint64_t kNone = ~0ull;
static_assert(kMaxRefs <= 16 && 4 + 1 + kCalBits + kCntBits == 64, "element layout");

__device__ __forceinline__ uint64_t find_key(uint32_t ref, uint32_t strand, int64_t cal) {
  return (static_cast<uint64_t>(ref) << (kCalBits + 1)) | (static_cast<uint64_t>(strand) << kCalBits) |
         static_cast<uint64_t>(cal + static_cast<int64_t>(kCalBias));
}

// a staged window of key K: start (low word, then the bits above 32 with the
// reference and strand), length, hits
__device__ __forceinline__ uint4 find_window(const FindArgs& a, uint64_t K, uint32_t m, uint32_t hits) {
  const uint32_t ref = static_cast<uint32_t>(K >> (kCalBits + 1));
  const uint32_t strand = static_cast<uint32_t>(K >> kCalBits) & 1u;
  const int64_t cal = static_cast<int64_t>(K & ((1ull << kCalBits) - 1)) - static_cast<int64_t>(kCalBias);
  const int64_t N = static_cast<int64_t>(a.di.ref_len[ref]);
  int64_t lo = cal - static_cast<int64_t>(a.pad), hi = cal + m + static_cast<int64_t>(a.pad);
  if (lo < 0) lo = 0;
  if (hi > N) hi = N;
  return make_uint4(static_cast<uint32_t>(lo), static_cast<uint32_t>(static_cast<uint64_t>(lo) >> 32) | (ref << 8) | (strand << 16),
                    static_cast<uint32_t>(hi - lo), hits);
}

// the CALs of entry e of reference r2 for a seed at so with orientation bits
// rori: the '+' one (or the only one) in *k1, true in *k1ok; a seed that is its
// own reverse complement may give both strands (then the '-' one in *k2)
__device__ __forceinline__ void entry_cals(const DevIndex& di, int r2, uint64_t e, uint32_t so, uint32_t rori, uint32_t m,
                                           uint64_t* k1, bool* ok1, uint64_t* k2, bool* ok2) {
  const uint32_t po = di.packed ? di.posor[r2][e] : 0u;
  const uint32_t fo = di.packed ? po >> 30 : di.orient[r2][e];
  const int64_t p = di.packed ? static_cast<int64_t>(po & 0x3fffffffu) : static_cast<int64_t>(di.pos[r2][e]);
  const bool plus = (fo & rori) != 0;
  const bool minus = ((fo & 1u) && (rori & 2u)) || ((fo & 2u) && (rori & 1u));
  const uint64_t km = find_key(r2, 1, p - static_cast<int64_t>(m - so - di.k));
  *k1 = plus ? find_key(r2, 0, p - so) : km;
  *ok1 = plus || minus;
  *k2 = km;
  *ok2 = plus && minus;
}

__device__ __forceinline__ bool bad_reads(const FindArgs& a) {
  return (*static_cast<volatile const uint32_t*>(a.status) & (kStBadRead | kStBadStart)) != 0;
}

constexpr int kFindWarps = 4;
constexpr uint32_t kRuns = 128;   // (CAL, count) runs a warp holds
constexpr uint32_t kRanks = 64;   // ranks it takes over a read's rounds and references
constexpr uint32_t kSlotChunk = 16;  // staging slots a warp takes at a time

struct WarpSpace {
  uint8_t q[kMaxReadLen];
  uint64_t el[kRuns];                // runs as found, then sorted
  unsigned long long best[kRuns];    // per window: (hits of its best CAL << 32) | ~element
  uint32_t pre[kRuns + 4];           // exclusive prefix of the elements' counts
  uint32_t wst[kRuns + 4];           // window starts, then the number of elements
  uint32_t pk[kPackWords], rk[kPackWords];
};

// sorts the nh elements of w.el (nh <= 32 E), merges them into windows; returns
// their number (starts in wst, best in best, count prefixes in pre)
template <int E>
__device__ __forceinline__ uint32_t warp_merge(WarpSpace& w, uint32_t nh, uint64_t merge_dist, int lane) {
  constexpr int P = 32 * E;
  const uint32_t le = (2u << lane) - 1u;  // lanes at or below this one (lane 31: all)
  uint64_t k[E];
#pragma unroll
  for (int h = 0; h < E; ++h) k[h] = 32u * h + lane < nh ? w.el[32 * h + lane] : kNone;
  // bitonic sort, ascending: the lower index of a pair keeps the minimum in
  // ascending runs ((e & size) == 0), the maximum in descending ones
  if (nh > 1) {
#pragma unroll
    for (int size = 2; size <= P; size <<= 1) {
#pragma unroll
      for (int stride = size / 2; stride > 0; stride >>= 1) {
        if (stride >= 32) {
          const int hs = stride / 32;
#pragma unroll
          for (int h = 0; h < E; ++h) {
            if (h & hs) continue;
            const bool up = ((32 * h + lane) & size) == 0;
            const uint64_t x = k[h], y = k[h | hs];
            if ((x > y) == up) {
              k[h] = y;
              k[h | hs] = x;
            }
          }
        } else {
#pragma unroll
          for (int h = 0; h < E; ++h) {
            const uint64_t y = __shfl_xor_sync(FULL, k[h], stride);
            const bool up = ((32 * h + lane) & size) == 0, low = (lane & stride) == 0;
            k[h] = (low == up) ? (k[h] < y ? k[h] : y) : (k[h] > y ? k[h] : y);
          }
        }
      }
    }
  }
  uint32_t total = 0;
#pragma unroll
  for (int h = 0; h < E; ++h) {
    const uint32_t e = 32 * h + lane;
    const uint32_t c = e < nh ? static_cast<uint32_t>(k[h]) & kCntMask : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    w.el[e] = k[h];
    w.pre[e] = total + x - c;
    total += __shfl_sync(FULL, x, 31);
  }
  if (lane == 0) w.pre[nh] = total;  // nh = P included: pre has room past P
  __syncwarp();
  // run starts (the CAL changes) and window starts ((ref, strand) changes or a
  // gap over merge_dist), as masks of the E groups of 32 elements
  uint32_t rm[E], wm[E];
  uint32_t nwin = 0;
#pragma unroll
  for (int h = 0; h < E; ++h) {
    const uint32_t e = 32 * h + lane;
    bool rs = false, ws = false;
    if (e < nh) {
      if (e == 0) {
        rs = ws = true;
      } else {
        const uint64_t p = w.el[e - 1] >> kCntBits, c = k[h] >> kCntBits;
        rs = c != p;
        ws = (c >> kCalBits) != (p >> kCalBits) || c - p > merge_dist;
      }
    }
    rm[h] = __ballot_sync(FULL, rs);
    wm[h] = __ballot_sync(FULL, ws);
    nwin += __popc(wm[h]);
  }
  for (uint32_t j = lane; j < nwin; j += 32) w.best[j] = 0ull;
  __syncwarp();
  uint32_t wbefore = 0;  // window starts in the groups before h
#pragma unroll
  for (int h = 0; h < E; ++h) {
    const uint32_t e = 32 * h + lane;
    if ((wm[h] >> lane) & 1u) w.wst[wbefore + __popc(wm[h] & (le >> 1))] = e;
    if ((rm[h] >> lane) & 1u) {
      const uint32_t win = wbefore + __popc(wm[h] & le) - 1u;  // the window holding this run
      uint32_t next = nh;                                      // the next run's start
      const uint32_t above = rm[h] & ~le;
      if (above) {
        next = 32 * h + __ffs(above) - 1;
      } else {
#pragma unroll
        for (int h2 = E - 1; h2 > h; --h2)
          if (rm[h2]) next = 32 * h2 + __ffs(rm[h2]) - 1;
      }
      // the most frequent CAL, the smallest of equally frequent ones
      const uint32_t hits = w.pre[next] - w.pre[e];
      atomicMax(&w.best[win], (static_cast<unsigned long long>(hits) << 32) | (0xffffffffu - e));
    }
    wbefore += __popc(wm[h]);
  }
  if (lane == 0) w.wst[nwin] = nh;
  __syncwarp();
  return nwin;
}

// What bounds it: random requests to the index, a seed's bucket head and its
// entry's position (300k reads of 100 bases against 2 x 16 Mbp: 45M of them in 0.81
// ms, 56 G/s, DRAM 72% busy; 2.36 warp instructions per cycle and SM).  So nothing but the
// lookups touches device memory, and the registers are held to 40 warps per SM to
// hide their latency.  1M such reads: 2.6 ms, where the count, emit, filter and
// compaction passes over kept lookups and CALs took 7.2 ms.  128 runs and 64
// ranks: a unique 250-base read has about 8 runs, and a read with more copies than
// that shares its counting better over a block.
__global__ void __launch_bounds__(32 * kFindWarps, 10) k_find_warp(FindArgs a) {
  __shared__ __align__(16) WarpSpace ws[kFindWarps];
  if (bad_reads(a)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpSpace& w = ws[warp];
  const int k = a.di.k;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t cap = min(kRuns, a.merge_keys);
  uint64_t slot = 0;
  uint32_t left = 0;  // staging slots this warp still holds
  for (uint32_t rr = blockIdx.x * kFindWarps + warp; rr < a.nr; rr += gridDim.x * kFindWarps) {
    const uint32_t r = a.r0 + rr;
    const uint64_t o0 = a.read_off[r];
    const uint32_t m = static_cast<uint32_t>(a.read_off[r + 1] - o0);
    uint32_t nh = 0, ranks = 0;
    bool bail = false;
    if (load_codes(a.bases, o0, m, w.q, lane, a.status) && m >= static_cast<uint32_t>(k)) {
      pack_codes(w.q, w.pk, w.rk, lane);
      uint64_t last = kNone;  // the CAL of the last run
      // one rank's CALs (of the lanes with ok) appended as runs
      auto append = [&](uint64_t K, bool ok) {
        const uint32_t mask = __ballot_sync(FULL, ok);
        if (!mask) return;
        const uint32_t below = mask & lt;
        uint64_t prev = __shfl_sync(FULL, K, below ? 31 - __clz(below) : lane);
        if (!below) prev = last;
        const bool head = ok && K != prev;
        const uint32_t hm = __ballot_sync(FULL, head);
        if (nh + __popc(hm) > cap) {
          bail = true;
          return;
        }
        const uint32_t lead = hm ? mask & ((1u << (__ffs(hm) - 1)) - 1u) : mask;  // still the last run's CAL
        if (lead && lane == 0) w.el[nh - 1] += __popc(lead);
        if (head) {
          const uint32_t above = hm & ~lt & ~(1u << lane);
          const uint32_t upto = above ? (1u << (__ffs(above) - 1)) - 1u : FULL;
          w.el[nh + __popc(hm & lt)] = (K << kCntBits) | __popc(mask & upto & ~lt);
        }
        nh += __popc(hm);
        last = __shfl_sync(FULL, K, 31 - __clz(mask));
        __syncwarp();
      };
      for (uint32_t o_base = 0; o_base + k <= m && !bail; o_base += 32 * a.stride) {
        const uint32_t o = o_base + lane * a.stride;
        const bool live = o + k <= m;
        // the seed's k-mer and its reverse complement's (at kMaxReadLen - o - k of
        // the padded reverse complement)
        const uint64_t fwd = live ? kmer_at(w.pk, o, k) : 0;
        const uint64_t rc = live ? kmer_at(w.rk, kMaxReadLen - o - k, k) : 0;
        const uint64_t canon = fwd < rc ? fwd : rc;
        const uint32_t rori = (fwd == canon ? 1u : 0u) | (rc == canon ? 2u : 0u);
        uint64_t pb = 0;
        uint32_t pkey = 0;
        uint32_t hl0 = 0, hh0 = 0, hl1 = 0, hh1 = 0;
        bool head = false;
        if (a.di.packed && live) {
          const int kb = 2 * (k - a.di.a);
          const uint64_t h = seed_hash(canon, k, a.di.hash_seed[0]);
          pb = h >> kb;
          pkey = static_cast<uint32_t>(h & mask_bits(kb));
          if (a.di.heads) head = lookup_head(a.di, pb, pkey, &hl0, &hh0, &hl1, &hh1);
        }
        for (int r2 = 0; r2 < a.di.n_refs && !bail; ++r2) {
          uint64_t lo = 0, hi = 0;
          if (live) {
            if (head) {
              lo = r2 ? hl1 : hl0;
              hi = r2 ? hh1 : hh0;
            } else if (a.di.packed) {
              lookup_packed(a.di, pb, pkey, r2, &lo, &hi);
            } else {
              lookup(a.di, r2, canon, &lo, &hi);
            }
          }
          const uint32_t cnt = static_cast<uint32_t>(hi - lo < kRanks + 1 ? hi - lo : kRanks + 1);
          const uint32_t most = __reduce_max_sync(FULL, cnt);
          ranks += most;
          if (ranks > kRanks) {
            bail = true;
            break;
          }
          for (uint32_t t = 0; t < most && !bail; ++t) {
            uint64_t k1 = 0, k2 = 0;
            bool ok1 = false, ok2 = false;
            if (t < cnt) entry_cals(a.di, r2, lo + t, o, rori, m, &k1, &ok1, &k2, &ok2);
            append(k1, ok1);
            if (!bail && __any_sync(FULL, ok2)) append(k2, ok2);
          }
        }
      }
    }
    uint32_t kept = 0;
    if (bail) {
      if (lane == 0) a.list_mid[atomicAdd(&a.plan->n_mid, 1u)] = rr;
    } else if (nh) {
      const uint32_t nwin = nh <= 32   ? warp_merge<1>(w, nh, a.merge_dist, lane)
                            : nh <= 64 ? warp_merge<2>(w, nh, a.merge_dist, lane)
                                       : warp_merge<4>(w, nh, a.merge_dist, lane);
      kept = a.max_cands && nwin > a.max_cands ? a.max_cands : nwin;
      if (left < kept) {
        left = kept > kSlotChunk ? kept : kSlotChunk;
        if (lane == 0) slot = atomicAdd(&a.plan->cursor, static_cast<unsigned long long>(left));
        slot = __shfl_sync(FULL, slot, 0);
      }
      const bool room = slot + kept <= a.win_cap;  // else the call is run again with more
      if (lane == 0) a.wslot[rr] = static_cast<uint32_t>(slot);
      uint32_t before = 0;
      for (uint32_t j0 = 0; j0 < nwin; j0 += 32) {
        const uint32_t j = j0 + lane;
        bool keep = j < nwin;
        const uint32_t hits = keep ? w.pre[w.wst[j + 1]] - w.pre[w.wst[j]] : 0u;
        if (kept < nwin && keep) {
          // the max_cands windows of most hits, the smaller key of equal ones, in key order
          uint32_t rank = 0;
          for (uint32_t q = 0; q < nwin; ++q) {
            const uint32_t hq = w.pre[w.wst[q + 1]] - w.pre[w.wst[q]];
            rank += (hq > hits || (hq == hits && q < j)) ? 1u : 0u;
          }
          keep = rank < a.max_cands;
        }
        const uint32_t km = __ballot_sync(FULL, keep);
        if (keep && room) {
          const uint32_t at = 0xffffffffu - static_cast<uint32_t>(w.best[j]);
          a.win[slot + before + __popc(km & lt)] = find_window(a, w.el[at] >> kCntBits, m, hits);
        }
        before += __popc(km);
      }
      slot += kept;
      left -= kept;
    }
    if (lane == 0) a.nwin[rr] = kept;
    __syncwarp();
  }
}

// One block per read.  S table slots (a power of two), up to 3/4 of them used; T
// threads; reads of more than ENTRIES entries are left to the larger block.
// Records of one reference's seeds at a time are taken by groups of eight lanes:
// most hold a few entries, a repeat's hold thousands, consecutive.  Bound by the
// shared-memory table (a load and an add per CAL) and, before reads of many
// entries went to the larger block, by the last small block's read.  10k reads of
// 250 bases, 30% repeats, no CAL limit (36M CALs, half of them of 294 reads with
// more than 16384): whole call 2.47 to 1.90 ms by that line (8192: 1.88, 32768:
// 2.04), 20k reads with limit 1024 1.94 to 1.40 (1.50, 1.78); 1.19 and 1.33 with
// 16384 instead of 8192 slots in the large table, which keeps reads like the one
// here of 8721 distinct CALs off the large-read path.  The small table leaves room
// for 10 blocks per SM.
// Reads of more distinct CALs than the large table takes cost about 0.5 ms each (the
// many-block path) where the table's cost 0.012 spread over the SMs (2000 reads in a
// repeat of 12,000 / 12,600 copies 23.0 / 1023 ms, 1035 / 1034 before the tables; one
// read 1.78 / 1.13 ms).  Cutting to max_cands takes each window's rank here, whatever
// their number (a look at max_cands every 256 windows; at each one, 20k reads cut to 64
// windows took 1302 us, 1289 so): 2000 reads of 12,000 windows 25.5 ms (1068 when more than
// 4096 windows went to the many-block path).
constexpr int kElBits = 14;  // bits of an element's number beside its count (at most one per seed)
constexpr uint32_t kElMask = (1u << kElBits) - 1u;
static_assert(2 * kMaxReadLen < (1 << (32 - kElBits)), "a CAL's count and an element number in 32 bits");

template <int S, int T, uint32_t ENTRIES>
struct BlockSpace {
  static constexpr uint32_t kDistinct = S / 4 * 3;
  static constexpr uint32_t kEntries = ENTRIES;
  // the table (keys, counts), then in its place the sorted elements (S) and each
  // window's best element and hits (kDistinct)
  static constexpr uint32_t kBytes = S * 8 + kDistinct * 8;
  static_assert(S <= (1 << kElBits), "element numbers");
};

template <int S, int T, uint32_t ENTRIES>
__global__ void __launch_bounds__(T) k_find_block(FindArgs a, const uint32_t* list, const uint32_t* n_list, uint32_t* queue,
                                                  uint32_t* next, uint32_t* n_next) {
  using Space = BlockSpace<S, T, ENTRIES>;
  constexpr int kGroup = 8, kGroups = T / kGroup, kPer = S / T;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ __align__(16) uint8_t q[kMaxReadLen];
  __shared__ uint32_t pk[kPackWords], rk[kPackWords];
  __shared__ uint64_t rec[kMaxReadLen];
  __shared__ uint32_t s_item, s_distinct, s_over, s_total;
  __shared__ unsigned long long s_slot;
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(sm);
  uint32_t* cnts = reinterpret_cast<uint32_t*>(sm + S * 8);
  uint64_t* el = reinterpret_cast<uint64_t*>(sm);
  uint32_t* best = reinterpret_cast<uint32_t*>(sm + S * 8);
  uint32_t* hits = best + Space::kDistinct;
  const uint32_t tid = threadIdx.x;
  const uint32_t most = min(Space::kDistinct, a.merge_keys);
  if (bad_reads(a)) return;
  const uint32_t n_items = *n_list;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(queue, 1u);
    __syncthreads();
    if (s_item >= n_items) return;
    const uint32_t rr = list[s_item], r = a.r0 + rr;
    const uint64_t o0 = a.read_off[r];
    const uint32_t m = static_cast<uint32_t>(a.read_off[r + 1] - o0);
    const int k = a.di.k;
    if (tid < 32) {
      load_codes(a.bases, o0, m, q, tid, a.status);
      pack_codes(q, pk, rk, tid);
    }
    for (uint32_t i = tid; i < S; i += T) {
      keys[i] = kNone;
      cnts[i] = 0;
    }
    if (tid == 0) {
      s_distinct = s_over = s_total = 0;
    }
    const uint32_t nseeds = (m - k) / a.stride + 1;  // listed reads have m >= k
    // one CAL into the table; past `most` distinct ones the read is given up (the
    // table still has room for one more per thread)
    auto insert = [&](uint64_t K) {
      uint32_t s = (static_cast<uint32_t>(K ^ (K >> 29)) * 2654435761u) >> (32 - __popc(S - 1));
      for (int probe = 0; probe < S; ++probe) {
        const uint64_t v = *reinterpret_cast<volatile unsigned long long*>(&keys[s]);
        if (v == K) break;
        if (v == kNone) {
          const uint64_t old = atomicCAS(&keys[s], kNone, K);
          if (old == kNone) {
            if (atomicAdd(&s_distinct, 1u) >= most) *static_cast<volatile uint32_t*>(&s_over) = 1;
            break;
          }
          if (old == K) break;
        }
        s = (s + 1) & (S - 1);
      }
      atomicAdd(&cnts[s], 1u);
    };
    for (int r2 = 0; r2 < a.di.n_refs; ++r2) {
      __syncthreads();
      if (s_over) break;  // written before the barrier only: the same for every thread
      __syncthreads();
      for (uint32_t si = tid; si < nseeds; si += T) {
        const uint32_t o = si * a.stride;
        const uint64_t fwd = kmer_at(pk, o, k), rc = kmer_at(rk, kMaxReadLen - o - k, k);
        const uint64_t canon = fwd < rc ? fwd : rc;
        const uint32_t rori = (fwd == canon ? 1u : 0u) | (rc == canon ? 2u : 0u);
        uint64_t lo = 0, hi = 0;
        if (a.di.packed) {
          const int kb = 2 * (k - a.di.a);
          const uint64_t h = seed_hash(canon, k, a.di.hash_seed[0]), pb = h >> kb;
          const uint32_t pkey = static_cast<uint32_t>(h & mask_bits(kb));
          uint32_t hl0 = 0, hh0 = 0, hl1 = 0, hh1 = 0;
          if (a.di.heads && lookup_head(a.di, pb, pkey, &hl0, &hh0, &hl1, &hh1)) {
            lo = r2 ? hl1 : hl0;
            hi = r2 ? hh1 : hh0;
          } else {
            lookup_packed(a.di, pb, pkey, r2, &lo, &hi);
          }
        } else {
          lookup(a.di, r2, canon, &lo, &hi);
        }
        // the entries of one key have distinct CALs: more of them than the table
        // takes need no counting
        const bool fits = hi - lo <= most && lo <= kRangeLoMax;
        if (!fits) s_over = 1;
        rec[si] = fits ? range_pack(lo, static_cast<uint32_t>(hi - lo), rori) : 0ull;
        if (fits && hi > lo) atomicAdd(&s_total, static_cast<uint32_t>(hi - lo));
      }
      __syncthreads();
      // too much work for this many threads: left to the larger block
      if (s_total > Space::kEntries) s_over = 1;
      __syncthreads();
      for (uint32_t si = tid / kGroup; si < nseeds; si += kGroups) {
        const uint64_t x = rec[si];
        const uint64_t lo = x >> 26;
        const uint32_t cnt = static_cast<uint32_t>(x >> 2) & kRangeCntMax, rori = static_cast<uint32_t>(x & 3u);
        for (uint32_t j = tid % kGroup; j < cnt; j += 4 * kGroup) {
          uint64_t k1[4], k2[4];
          bool ok1[4], ok2[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            ok1[u] = ok2[u] = false;
            if (j + u * kGroup < cnt)
              entry_cals(a.di, r2, lo + j + u * kGroup, si * a.stride, rori, m, &k1[u], &ok1[u], &k2[u], &ok2[u]);
          }
          if (*static_cast<volatile uint32_t*>(&s_over)) break;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (ok1[u] && !*static_cast<volatile uint32_t*>(&s_over)) insert(k1[u]);
            if (ok2[u] && !*static_cast<volatile uint32_t*>(&s_over)) insert(k2[u]);
          }
        }
      }
    }
    __syncthreads();
    if (s_over || s_distinct > most) {
      if (tid == 0) next[atomicAdd(n_next, 1u)] = rr;
      if (tid == 0) a.nwin[rr] = 0;
      __syncthreads();
      continue;
    }
    // the distinct CALs with their counts, packed and sorted
    uint64_t mine[kPer];
    uint32_t have = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const uint64_t K = keys[tid * kPer + u];
      mine[u] = K == kNone ? kNone : (K << kCntBits) | cnts[tid * kPer + u];
      have += K == kNone ? 0u : 1u;
    }
    uint64_t tot = 0;
    uint32_t at = static_cast<uint32_t>(block_exscan(have, &tot));  // a barrier inside: the table is read
    const uint32_t n = static_cast<uint32_t>(tot);
#pragma unroll
    for (int u = 0; u < kPer; ++u)
      if (mine[u] != kNone) el[at++] = mine[u];
    const uint32_t P = pow2_at_least(n);
    for (uint32_t i = n + tid; i < P; i += T) el[i] = kNone;
    __syncthreads();
    bitonic(el, P);
    // windows, their starts numbered by a prefix sum over the threads' slices; each
    // slice offers its part of a window its most frequent CAL (the smallest of
    // equally frequent ones) and adds its hits
    const uint32_t per = (n + T - 1) / T, i0 = min(n, tid * per), i1 = min(n, i0 + per);
    auto starts = [&](uint32_t i) {
      if (i == 0) return true;
      const uint64_t c = el[i] >> kCntBits, p = el[i - 1] >> kCntBits;
      return (c >> kCalBits) != (p >> kCalBits) || c - p > static_cast<uint64_t>(a.merge_dist);
    };
    uint32_t sum = 0;
    for (uint32_t i = i0; i < i1; ++i) sum += starts(i) ? 1u : 0u;
    uint32_t wk = static_cast<uint32_t>(block_exscan(sum, &tot));
    const uint32_t nwin = static_cast<uint32_t>(tot);
    for (uint32_t j = tid; j < nwin; j += T) best[j] = hits[j] = 0;
    __syncthreads();
    {
      uint32_t top = 0, add = 0;
      for (uint32_t i = i0; i < i1; ++i) {
        if (starts(i)) {
          if (add) {
            atomicMax(&best[wk - 1], top);
            atomicAdd(&hits[wk - 1], add);
          }
          top = add = 0;
          ++wk;
        }
        const uint32_t c = static_cast<uint32_t>(el[i]) & kCntMask;
        top = max(top, (c << kElBits) | (kElMask - i));
        add += c;
      }
      if (add) {
        atomicMax(&best[wk - 1], top);
        atomicAdd(&hits[wk - 1], add);
      }
    }
    __syncthreads();
    const bool cut = a.max_cands && nwin > a.max_cands;
    const uint32_t kept = cut ? a.max_cands : nwin;
    if (tid == 0) {
      s_slot = atomicAdd(&a.plan->cursor, static_cast<unsigned long long>(kept));
      a.wslot[rr] = static_cast<uint32_t>(s_slot);
      a.nwin[rr] = kept;
    }
    __syncthreads();
    const bool room = s_slot + kept <= a.win_cap;
    uint32_t before = 0;
    for (uint32_t j0 = 0; j0 < nwin; j0 += T) {
      const uint32_t j = j0 + tid;
      uint32_t at = j;
      bool keep = j < nwin;
      if (cut) {
        // the max_cands windows of most hits, the smaller key of equal ones, in key order
        if (keep) {
          uint32_t rank = 0;
          const uint32_t h = hits[j];
          for (uint32_t q1 = 0; q1 < nwin && rank < a.max_cands; q1 += 256) {
            const uint32_t end = min(nwin, q1 + 256);
            for (uint32_t q2 = q1; q2 < end; ++q2) rank += (hits[q2] > h || (hits[q2] == h && q2 < j)) ? 1u : 0u;
          }
          keep = rank < a.max_cands;
        }
        at = before + static_cast<uint32_t>(block_exscan(keep ? 1u : 0u, &tot));
        before += static_cast<uint32_t>(tot);
      }
      if (keep && room) a.win[s_slot + at] = find_window(a, el[kElMask - (best[j] & kElMask)] >> kCntBits, m, hits[j]);
    }
    __syncthreads();
  }
}

// offsets of device reads: decreasing ones, reads over kMaxReadLen bases, a
// first offset that is not 0 (the finder's kernels read nothing after one)
__global__ void k_find_check(const uint64_t* off, uint32_t n, uint32_t* status) {
  const uint64_t r = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x;
  if (r == 0 && off[0] != 0) atomicOr(status, kStBadStart);
  if (r < n && (off[r + 1] < off[r] || off[r + 1] - off[r] > static_cast<uint64_t>(kMaxReadLen))) atomicOr(status, kStBadRead);
}

// The windows of reads r0 .. r0 + nr from the staging area to the list: one
// thread per window (its read by binary search of the offsets, whose top levels
// stay in L1), so reads of thousands of windows cost no more per window than
// reads of one; the first nr + 1 threads also write the list's offsets.
__global__ void k_find_out(const uint64_t* woff, uint32_t nr, uint64_t nw, const uint32_t* wslot, const uint4* win,
                           uint64_t base, FindList l) {
  const uint64_t i = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x;
  if (i <= nr) l.off[i] = base + woff[i];
  if (i >= nw) return;
  uint32_t lo = 0, hi = nr;  // the last read whose first window is at or before i
  while (lo + 1 < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (woff[mid] <= i) lo = mid;
    else hi = mid;
  }
  const uint4 x = win[wslot[lo] + (i - woff[lo])];
  const uint64_t d = base + i;
  l.ref[d] = static_cast<uint8_t>(x.y >> 8);
  l.strand[d] = static_cast<uint8_t>(x.y >> 16);
  l.start[d] = x.x | (static_cast<uint64_t>(x.y & 0xffu) << 32);
  l.len[d] = x.z;
  l.hits[d] = x.w;
}

// the reads listed for the large-read path as a batch of their own: their
// lengths (a scan makes offsets of them), then their bases
__global__ void k_rest_len(const uint64_t* off, uint32_t r0, const uint32_t* list, uint32_t n, uint32_t* len) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) len[i] = static_cast<uint32_t>(off[r0 + list[i] + 1] - off[r0 + list[i]]);
}

__global__ void k_rest_bases(const char* bases, const uint64_t* off, uint32_t r0, const uint32_t* list, uint32_t n,
                             const uint64_t* noff, char* out) {
  const uint32_t i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (i >= n) return;
  const uint64_t o = off[r0 + list[i]];
  for (uint32_t t = threadIdx.x & 31; t < noff[i + 1] - noff[i]; t += 32) out[noff[i] + t] = bases[o + t];
}

// the large-read path's list back into the staging area from slot `base`
__global__ void k_rest_stage(FindList l, const uint32_t* list, uint32_t n, uint64_t base, uint4* win, uint32_t* nwin,
                             uint32_t* wslot) {
  const uint32_t i = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (i >= n) return;
  const uint64_t b0 = l.off[i], b1 = l.off[i + 1];
  for (uint64_t t = b0 + (threadIdx.x & 31); t < b1; t += 32)
    win[base + t] = make_uint4(static_cast<uint32_t>(l.start[t]),
                               static_cast<uint32_t>(l.start[t] >> 32) | (static_cast<uint32_t>(l.ref[t]) << 8) |
                                   (static_cast<uint32_t>(l.strand[t]) << 16),
                               l.len[t], l.hits[t]);
  if ((threadIdx.x & 31) == 0) {
    nwin[list[i]] = static_cast<uint32_t>(b1 - b0);
    wslot[list[i]] = static_cast<uint32_t>(base + b0);
  }
}

constexpr int kMidS = 1024, kMidT = 128, kWideS = 16384, kWideT = 1024;
constexpr uint32_t kMidEntries = 16384, kWideEntries = 0xffffffffu;
using MidSpace = BlockSpace<kMidS, kMidT, kMidEntries>;
using WideSpace = BlockSpace<kWideS, kWideT, kWideEntries>;

}  // namespace

int launch_find_check(const uint64_t* read_off, uint32_t n, uint32_t* status, cudaStream_t st) {
  k_find_check<<<n / 256 + 1, 256, 0, st>>>(read_off, n, status);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_find(const FindArgs& a, cudaStream_t st) {
  if (a.nr == 0) return 0;
  // per device, so set for each launch
  if (cudaFuncSetAttribute(k_find_block<kWideS, kWideT, kWideEntries>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(WideSpace::kBytes)) != cudaSuccess)
    return -1;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  auto grid = [&](uint32_t per_block, uint32_t blocks_per_sm) {
    const uint32_t need = (a.nr + per_block - 1) / per_block, most = static_cast<uint32_t>(nsm) * blocks_per_sm;
    return need < most ? need : most;
  };
  k_find_warp<<<grid(kFindWarps, 40), 32 * kFindWarps, 0, st>>>(a);
  k_find_block<kMidS, kMidT, kMidEntries><<<grid(1, 10), kMidT, MidSpace::kBytes, st>>>(a, a.list_mid, &a.plan->n_mid, &a.plan->q_mid,
                                                                         a.list_wide, &a.plan->n_wide);
  k_find_block<kWideS, kWideT, kWideEntries><<<grid(1, 1), kWideT, WideSpace::kBytes, st>>>(a, a.list_wide, &a.plan->n_wide,
                                                                             &a.plan->q_wide, a.list_rest, &a.plan->n_rest);
  return cudaPeekAtLastError() == cudaSuccess ? 3 : -1;
}

int launch_find_out(const uint64_t* woff, uint32_t nr, uint64_t nw, const uint32_t* wslot, const uint4* win, uint64_t base,
                    const FindList& l, cudaStream_t st) {
  const uint64_t n = nw > nr ? nw : nr + 1ull;
  k_find_out<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(woff, nr, nw, wslot, win, base, l);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int launch_rest_gather(const char* bases, const uint64_t* read_off, uint32_t r0, const uint32_t* list, uint32_t n,
                       uint32_t* len, uint64_t* off, uint64_t* sums, char* out, cudaStream_t st) {
  if (n == 0) return 0;
  k_rest_len<<<(n + 255) / 256, 256, 0, st>>>(read_off, r0, list, n, len);
  if (launch_scan_u64(len, n, off, sums, st) < 0) return -1;
  k_rest_bases<<<(n + 7) / 8, 256, 0, st>>>(bases, read_off, r0, list, n, off, out);
  return cudaPeekAtLastError() == cudaSuccess ? 5 : -1;
}

int launch_rest_stage(const FindList& l, const uint32_t* list, uint32_t n, uint64_t base, uint4* win, uint32_t* nwin,
                      uint32_t* wslot, cudaStream_t st) {
  if (n == 0) return 0;
  k_rest_stage<<<(n + 7) / 8, 256, 0, st>>>(l, list, n, base, win, nwin, wslot);
  return cudaPeekAtLastError() == cudaSuccess ? 1 : -1;
}

int preload_find() {
  int n_ = 0;
  SR_TOUCH(k_find_check);
  SR_TOUCH(k_find_warp);
  SR_TOUCH((k_find_block<kMidS, kMidT, kMidEntries>));
  SR_TOUCH((k_find_block<kWideS, kWideT, kWideEntries>));
  SR_TOUCH(k_find_out);
  SR_TOUCH(k_rest_len);
  SR_TOUCH(k_rest_bases);
  SR_TOUCH(k_rest_stage);
  return n_;
}

}  // namespace sr
