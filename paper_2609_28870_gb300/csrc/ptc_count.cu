// Stage c on a trace without runs: the stack distance of every access by
// counting, with no matrix and no queries.
//
// With r(i) = re-reads before access i, a re-read i with p = prev[i] has
//   SD_i = #{ j < i : v_j < v_i } - p,   v = prev + 1, none -> 0
//        = (i - r(i)) + #{ re-reads j < i : prev[j] < p } - p,
// because every first access before i has v = 0.  Read the re-reads in the
// order of prev (position p of the trace holds the re-read next[p]): the count
// is then the number of earlier entries of that sequence with a smaller rank
// r, and the ranks of M re-reads are a permutation of 0 .. M - 1.
//
// Counting the smaller entries before each entry of a permutation is a radix
// partition from the top digit down that keeps order: an entry counts, at each
// level, the earlier entries of its node with a smaller digit, and then moves
// to its digit's child node.  A node of 2^s ranks holds exactly 2^s entries
// and starts at a multiple of 2^s, so no node needs a table.  Two levels:
//   across buckets of 2^15 ranks, through global memory
//     k_cnt_next    next[] (scatter) and the bitmap of re-reads
//     (bitmap_ranks)  ranks before every word of it, and M
//     k_cnt_rank    rank of every entry, and bucket counts per tile
//     k_cnt_rows    their prefixes over the tiles, one CTA per bucket
//     k_cnt_scatter every entry: entries of smaller buckets before it (tiles
//                   before its own from the prefixes, its tile's by sorting
//                   the tile), and its low 15 bits to its bucket, in order
//   inside a bucket, in shared memory
//     k_cnt_bucket  three levels of radix 32: ballots count the smaller
//                   digits inside 32 entries, a running count per digit (one
//                   digit per lane) those before them
//   k_cnt_out       distances in access order
// Every pass streams; bound by instruction issue in the scatter and bucket
// kernels (about 70 instructions per 32 entries and level).  The matrix over
// every access (ptc_wavelet.cu) spent its time on one walk of 24 levels, two
// random sectors each, per access: 12M accesses of a block trace took 3.6 ms
// there and 0.53 ms here.
//
// Up to kCntMaxBuckets buckets (33.5M re-reads).  prev must take each value at
// most once; if it does not, next[] holds fewer entries than there are
// re-reads, the kernels after k_cnt_rank stop and the caller falls back to the
// matrix.
#include "ptc_internal.h"

namespace ptc {
namespace {

constexpr uint32_t kCntBucketLog2 = 15;
constexpr uint32_t kCntBucket = 1u << kCntBucketLog2;
constexpr uint32_t kCntMaxBuckets = 1023;  // and one digit for the positions without a next use
constexpr uint32_t kCntDigits = 1024;
constexpr int kCntThreads = 256;
constexpr int kCntWarps = kCntThreads / 32;
constexpr uint32_t kCntWarpTile = 1024;                    // positions per warp: 32 rounds of 32
constexpr uint32_t kCntTile = kCntWarps * kCntWarpTile;    // 8,192

// The digits of 32 entries, one per lane, seen two ways: the lanes whose digit
// is below / equal to this lane's own digit, and those whose digit is below /
// equal to the lane's number.
struct DigitMasks {
  uint32_t below, same, below_lane, at_lane;
};
__device__ __forceinline__ DigitMasks digit_masks(uint32_t d, uint32_t lane) {
  DigitMasks m{0, kFull, 0, kFull};
#pragma unroll
  for (int b = 4; b >= 0; --b) {
    const uint32_t ones = __ballot_sync(kFull, (d >> b) & 1u);
    if ((d >> b) & 1u) {
      m.below |= m.same & ~ones;
      m.same &= ones;
    } else {
      m.same &= ~ones;
    }
    if ((lane >> b) & 1u) {
      m.below_lane |= m.at_lane & ~ones;
      m.at_lane &= ones;
    } else {
      m.at_lane &= ~ones;
    }
  }
  return m;
}

// One warp, a node of 1,024 ranks in `it`: item = rank (10 bits, all of 0 ..
// 1023 present) plus a count from bit kShift up.  Leaves at it[rank] the item
// of that rank with the smaller ranks before it added to its count.
template <int kShift>
__device__ __forceinline__ void count_1024(uint32_t* it, uint32_t lane) {
  uint32_t x[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) x[c] = it[32 * c + lane];
  __syncwarp();
  uint32_t at = 0, below = 0;  // entries so far with digit = lane, and with digit < lane
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const uint32_t d = (x[c] >> 5) & 31u;
    const DigitMasks m = digit_masks(d, lane);
    const uint32_t smaller = __shfl_sync(kFull, below, d) + __popc(m.below & lanemask_lt());
    const uint32_t place = __shfl_sync(kFull, at, d) + __popc(m.same & lanemask_lt());
    it[32 * d + place] = x[c] + (smaller << kShift);
    at += __popc(m.at_lane);
    below += __popc(m.below_lane);
  }
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 32; ++c) x[c] = it[32 * c + lane];
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const uint32_t d = x[c] & 31u;
    const DigitMasks m = digit_masks(d, lane);
    it[32 * c + d] = x[c] + (__popc(m.below & lanemask_lt()) << kShift);
  }
  __syncwarp();
}

struct CountArgs {
  const uint32_t* prev;
  uint32_t n, T, buckets;   // buckets: an upper bound from n
  uint32_t* next;           // position -> its next use (kNone without one)
  uint32_t* rbits;          // re-read bitmap over accesses
  const uint32_t* rpre;     // re-reads before every word of it
  uint32_t* rank;           // position -> rank of its next use (kNone without one)
  uint32_t *cnt, *off;      // per bucket and tile: entries, and those of the tiles before
  uint16_t* low;            // entries of every bucket in order: low 15 bits of the rank
  uint32_t* acc;            // per rank: smaller ranks before it
  uint32_t* dist;
  const uint64_t* m;        // re-reads
  uint32_t* found;          // positions with a next use
  DevStatus* st;
};

// Whether prev took each value at most once (checked after k_cnt_rank).
__device__ __forceinline__ bool count_ok(const CountArgs& a) { return *a.m == (uint64_t)*a.found; }

__global__ void __launch_bounds__(256) k_cnt_next(CountArgs a) {
  grid_dep_sync();
  const uint32_t base = blockIdx.x * 2048 + threadIdx.x;
  uint32_t p[8];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 8; ++k) p[k] = base + 256 * k < a.n ? __ldcs(&a.prev[base + 256 * k]) : kNone;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t i = base + 256 * k;
    if (p[k] != kNone) {
      if (p[k] < i)
        a.next[p[k]] = i;
      else
        bad = true;
    }
    const uint32_t w = __ballot_sync(kFull, p[k] != kNone);
    if ((threadIdx.x & 31) == 0 && i < a.n) a.rbits[i >> 5] = w;
  }
  if (bad) raise_err(a.st, kErrInvalid);
}

__global__ void __launch_bounds__(kCntThreads) k_cnt_rank(CountArgs a) {
  grid_dep_sync();
  __shared__ uint32_t s_cnt[kCntDigits];
  __shared__ uint32_t s_found;
  for (uint32_t d = threadIdx.x; d < kCntDigits; d += kCntThreads) s_cnt[d] = 0;
  if (threadIdx.x == 0) s_found = 0;
  __syncthreads();
  const uint32_t base = blockIdx.x * kCntTile + threadIdx.x;
  uint32_t mine = 0;
  for (uint32_t k0 = 0; k0 < kCntTile; k0 += 8 * kCntThreads) {
    uint32_t i[8], r[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t p = base + k0 + kCntThreads * k;
      i[k] = p < a.n ? a.next[p] : kNone;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      r[k] = i[k] != kNone ? a.rpre[i[k] >> 5] + __popc(a.rbits[i[k] >> 5] & ((1u << (i[k] & 31)) - 1u)) : kNone;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t p = base + k0 + kCntThreads * k;
      if (p < a.n) a.rank[p] = r[k];
      if (r[k] != kNone) {
        ++mine;
        atomicAdd(&s_cnt[r[k] >> kCntBucketLog2], 1u);
      }
    }
  }
  mine = __reduce_add_sync(kFull, mine);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_found, mine);
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < a.buckets; d += kCntThreads) a.cnt[(size_t)d * a.T + blockIdx.x] = s_cnt[d];
  if (threadIdx.x == 0 && s_found) atomicAdd(a.found, s_found);
}

// One CTA per bucket: off[d][t] = cnt[d][0] + ... + cnt[d][t - 1].
__global__ void __launch_bounds__(kCntThreads) k_cnt_rows(CountArgs a) {
  grid_dep_sync();
  __shared__ uint32_t s_w[kCntWarps];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t* row = a.cnt + (size_t)blockIdx.x * a.T;
  uint32_t* out = a.off + (size_t)blockIdx.x * a.T;
  uint32_t run = 0;
  for (uint32_t t0 = 0; t0 < a.T; t0 += kCntThreads) {
    const uint32_t t = t0 + threadIdx.x;
    const uint32_t c = t < a.T ? row[t] : 0u;
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int ww = 0; ww < kCntWarps; ++ww) {
      before += ww < (int)w ? s_w[ww] : 0u;
      all += s_w[ww];
    }
    if (t < a.T) out[t] = run + before + x - c;
    run += all;
    __syncthreads();
  }
}

// Exclusive prefix over the 1,024 entries of `v` in place, by one warp.
template <class V>
__device__ __forceinline__ void warp_prefix_1024(V* v, uint32_t lane) {
  uint32_t run = 0;
#pragma unroll 4
  for (int j = 0; j < 32; ++j) {
    const uint32_t c = v[32 * j + lane];
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    v[32 * j + lane] = (V)(run + x - c);
    run += __shfl_sync(kFull, x, 31);
  }
  __syncwarp();
}

struct ScatterSmem {
  uint32_t item[kCntTile];                  // per warp: places among its 1,024 positions, with counts
  uint16_t place[kCntTile];                 // per position: its place in the warp's order
  uint16_t num[kCntWarps][kCntDigits];      // entries of each digit per warp, then in the warps before
  uint16_t start[kCntWarps][kCntDigits];    // entries of smaller digits in the warp, then in the warps before
  uint32_t off[kCntDigits];                 // entries of each digit in the tiles before
  uint32_t less[kCntDigits];                // entries of smaller digits in the tiles before
};

__device__ __forceinline__ uint32_t bucket_of(uint32_t r) {
  return r != kNone ? r >> kCntBucketLog2 : kCntDigits - 1;
}

// A tile of 8,192 positions, 1,024 per warp.  A warp orders its positions by
// (bucket, position), positions without a next use last; the places in that
// order are a permutation of 0 .. 1023, for which count_1024 gives each entry
// the entries of smaller buckets and the earlier ones of its own bucket before
// it in the warp.  The tables give those of the warps and the tiles before.
// The ranks are read three times (from L2) rather than kept, so that two CTAs
// fit an SM.
__global__ void __launch_bounds__(kCntThreads, 2) k_cnt_scatter(CountArgs a) {
  grid_dep_sync();
  extern __shared__ unsigned char s_raw[];
  ScatterSmem& S = *reinterpret_cast<ScatterSmem*>(s_raw);
  if (!count_ok(a)) return;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, tile = blockIdx.x;
  for (uint32_t d = threadIdx.x; d < kCntDigits; d += kCntThreads) {
    const uint32_t o = d < a.buckets ? a.off[(size_t)d * a.T + tile] : 0u;
    S.off[d] = o;
    S.less[d] = o;
#pragma unroll
    for (int ww = 0; ww < kCntWarps; ++ww) S.num[ww][d] = 0;
  }
  __syncthreads();
  uint16_t* num = S.num[w];
  uint16_t* start = S.start[w];
  uint32_t* item = S.item + w * kCntWarpTile;
  uint16_t* place = S.place + w * kCntWarpTile;
  const uint32_t p0 = tile * kCntTile + w * kCntWarpTile + lane;
  // earlier entries of the same digit in the warp
  for (int c0 = 0; c0 < 32; c0 += 8) {
    uint32_t r[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) r[c] = p0 + 32 * (c0 + c) < a.n ? a.rank[p0 + 32 * (c0 + c)] : kNone;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t d = bucket_of(r[c]);
      const uint32_t peers = __match_any_sync(kFull, d);
      const uint32_t same = num[d] + __popc(peers & lanemask_lt());
      __syncwarp();
      if ((peers & lanemask_lt()) == 0) num[d] = (uint16_t)(same + __popc(peers));
      place[32 * (c0 + c) + lane] = (uint16_t)same;
      __syncwarp();
    }
  }
  for (uint32_t d = lane; d < kCntDigits; d += 32) start[d] = num[d];
  __syncwarp();
  warp_prefix_1024(start, lane);
  for (int c0 = 0; c0 < 32; c0 += 8) {
    uint32_t r[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) r[c] = p0 + 32 * (c0 + c) < a.n ? a.rank[p0 + 32 * (c0 + c)] : kNone;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t x = 32 * (c0 + c) + lane, q = start[bucket_of(r[c])] + place[x];
      place[x] = (uint16_t)q;
      item[x] = q;
    }
  }
  __syncwarp();
  count_1024<10>(item, lane);
  if (w == 0) warp_prefix_1024(S.less, lane);
  // (earlier entries of the same bucket) | (of smaller buckets) << 16 in the
  // warp, while `start` still holds the warp's own prefixes
  uint32_t both[32];
#pragma unroll
  for (int c0 = 0; c0 < 32; c0 += 8) {
    uint32_t r[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) r[c] = p0 + 32 * (c0 + c) < a.n ? a.rank[p0 + 32 * (c0 + c)] : kNone;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint32_t q = place[32 * (c0 + c) + lane], same = q - start[bucket_of(r[c])];
      both[c0 + c] = same | ((item[q] >> 10) - same) << 16;
    }
  }
  __syncthreads();
  for (uint32_t d = threadIdx.x; d < kCntDigits; d += kCntThreads) {
    uint32_t x = 0, y = 0;
#pragma unroll
    for (int ww = 0; ww < kCntWarps; ++ww) {
      const uint32_t u = S.num[ww][d], v = S.start[ww][d];
      S.num[ww][d] = (uint16_t)x;
      S.start[ww][d] = (uint16_t)y;
      x += u;
      y += v;
    }
  }
  __syncthreads();
  const uint32_t m = (uint32_t)*a.m;
#pragma unroll
  for (int c0 = 0; c0 < 32; c0 += 8) {
    uint32_t r[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) r[c] = p0 + 32 * (c0 + c) < a.n ? a.rank[p0 + 32 * (c0 + c)] : kNone;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (r[c] == kNone) continue;
      const uint32_t d = r[c] >> kCntBucketLog2;
      const uint32_t dst = d * kCntBucket + S.off[d] + num[d] + (both[c0 + c] & 0xFFFFu);
      if (in_bounds(a.st, dst, m) && in_bounds(a.st, r[c], m)) {
        a.low[dst] = (uint16_t)(r[c] & (kCntBucket - 1));
        a.acc[r[c]] = S.less[d] + start[d] + (both[c0 + c] >> 16);
      }
    }
  }
}

// One bucket of 2^15 ranks in shared memory (item = rank, 15 bits, plus the
// count above them): a level of radix 32 across the CTA's 32 warps, then two
// inside each warp's 1,024.  A last bucket that is not full is padded with its
// missing ranks at the end, which no entry counts.
__global__ void __launch_bounds__(1024) k_cnt_bucket(CountArgs a) {
  grid_dep_sync();
  extern __shared__ unsigned char s_raw[];
  uint32_t* item = reinterpret_cast<uint32_t*>(s_raw);
  __shared__ uint32_t s_tab[32][33];
  const uint64_t M = *a.m;
  const uint64_t r0 = (uint64_t)blockIdx.x * kCntBucket;
  if (r0 >= M || !count_ok(a)) return;
  const uint32_t size = M - r0 < kCntBucket ? (uint32_t)(M - r0) : kCntBucket;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t at = 0;
#pragma unroll 8
  for (int c = 0; c < 32; ++c) {
    const uint32_t x = w * 1024 + 32 * c + lane;
    const uint32_t d = (x < size ? (uint32_t)__ldg(&a.low[r0 + x]) : x) >> 10;
    at += __popc(digit_masks(d, lane).at_lane);
  }
  s_tab[w][lane] = at;
  __syncthreads();
  {  // entries of digit w in the warps before `lane`
    const uint32_t c = s_tab[lane][w];
    uint32_t x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    s_tab[lane][w] = x - c;
  }
  __syncthreads();
  at = s_tab[w][lane];
  uint32_t below = at;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, below, o);
    if (lane >= (uint32_t)o) below += y;
  }
  below -= at;
#pragma unroll 8
  for (int c = 0; c < 32; ++c) {
    const uint32_t x = w * 1024 + 32 * c + lane;
    const uint32_t v = x < size ? (uint32_t)__ldg(&a.low[r0 + x]) : x;
    const uint32_t d = v >> 10;
    const DigitMasks m = digit_masks(d, lane);
    const uint32_t smaller = __shfl_sync(kFull, below, d) + __popc(m.below & lanemask_lt());
    const uint32_t place = __shfl_sync(kFull, at, d) + __popc(m.same & lanemask_lt());
    item[1024 * d + place] = v + (smaller << 15);
    at += __popc(m.at_lane);
    below += __popc(m.below_lane);
  }
  __syncthreads();
  uint32_t* mine = item + w * 1024;
  count_1024<15>(mine, lane);
#pragma unroll 8
  for (int c = 0; c < 32; ++c) {
    const uint32_t x = w * 1024 + 32 * c + lane;
    if (x < size) a.acc[r0 + x] += mine[32 * c + lane] >> 15;
  }
}

__global__ void __launch_bounds__(256) k_cnt_out(CountArgs a) {
  grid_dep_sync();
  if (!count_ok(a)) return;
  const uint32_t base = blockIdx.x * 2048 + threadIdx.x;
  uint32_t p[8], r[8], c[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t i = base + 256 * k;
    p[k] = i < a.n ? __ldcs(&a.prev[i]) : kNone;
    r[k] = i < a.n ? a.rpre[i >> 5] + __popc(a.rbits[i >> 5] & lanemask_lt()) : 0u;
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) c[k] = p[k] != kNone ? __ldcs(&a.acc[r[k]]) : 0u;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t i = base + 256 * k;
    if (i < a.n) __stcs(&a.dist[i], p[k] != kNone ? (i - r[k]) + c[k] - p[k] : kNone);
  }
}

struct CountLayout {
  DevStatus* st;
  uint32_t* done;
  uint32_t* found;
  size_t zero_bytes;
  uint64_t* m;
  uint32_t *next, *rank;
  uint32_t *rbits, *rpre, *tcnt, *tpre;
  uint32_t *cnt, *off;
  uint32_t* acc;
  uint16_t* low;
  uint32_t nwords, T, buckets;
  size_t total;
};

CountLayout count_layout(void* ws, uint64_t n) {
  CountLayout L;
  Carver cv(ws);
  const uint64_t nn = n ? n : 1;
  L.nwords = ceil_div_u32(nn, 32);
  L.T = ceil_div_u32(nn, kCntTile);
  L.buckets = ceil_div_u32(nn, kCntBucket);
  L.st = cv.take<DevStatus>(1);
  L.done = cv.take<uint32_t>(1);
  L.found = cv.take<uint32_t>(1);
  L.zero_bytes = cv.off;
  L.m = cv.take<uint64_t>(1);
  L.next = cv.take<uint32_t>(nn);
  L.rank = cv.take<uint32_t>(nn);
  L.rbits = cv.take<uint32_t>(L.nwords + 1);
  L.rpre = cv.take<uint32_t>(L.nwords + 1);
  L.tcnt = cv.take<uint32_t>(rank_tiles(L.nwords) + 1);
  L.tpre = cv.take<uint32_t>(rank_tiles(L.nwords) + 1);
  L.cnt = cv.take<uint32_t>((size_t)L.buckets * L.T);
  L.off = cv.take<uint32_t>((size_t)L.buckets * L.T);
  L.acc = cv.take<uint32_t>(nn);
  L.low = cv.take<uint16_t>((size_t)L.buckets * kCntBucket);
  L.total = cv.bytes();
  return L;
}

}  // namespace

bool stack_distance_countable(uint64_t n) { return n <= (uint64_t)kCntMaxBuckets * kCntBucket; }

size_t stack_distance_count_bytes(uint64_t n) {
  return stack_distance_countable(n) ? count_layout(nullptr, n).total : 0;
}

ptc_status stack_distance_count(const uint32_t* prev, uint64_t n, uint32_t* dist_out, void* ws, size_t ws_bytes,
                                cudaStream_t s, bool* counted) {
  *counted = false;
  if (!stack_distance_countable(n)) return PTC_ERR_INVALID_ARG;
  const CountLayout L = count_layout(ws, n);
  if (!ws_ok(ws, ws_bytes, L.total)) return PTC_ERR_WORKSPACE;
  const FillRange zf[2] = {{ws, L.zero_bytes, 0u}, {L.next, sizeof(uint32_t) * n, ~0u}};
  if (fill_many_async(zf, 2, s) != PTC_OK) return PTC_ERR_CUDA;
  if (cudaFuncSetAttribute(k_cnt_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ScatterSmem)) !=
          cudaSuccess ||
      cudaFuncSetAttribute(k_cnt_bucket, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(sizeof(uint32_t) * kCntBucket)) != cudaSuccess)
    return PTC_ERR_CUDA;
  const CountArgs a{prev, (uint32_t)n, L.T, L.buckets, L.next, L.rbits, L.rpre, L.rank, L.cnt, L.off, L.low, L.acc,
                    dist_out, L.m, L.found, L.st};
  PTC_KERNEL("k_cnt_next", s, k_cnt_next, ceil_div_u32(n, 2048), 256, 0, a);
  if (bitmap_ranks(L.rbits, L.nwords, L.rpre, L.tcnt, L.tpre, L.done, L.m, s) != PTC_OK) return PTC_ERR_CUDA;
  PTC_KERNEL("k_cnt_rank", s, k_cnt_rank, L.T, kCntThreads, 0, a);
  PTC_KERNEL("k_cnt_rows", s, k_cnt_rows, L.buckets, kCntThreads, 0, a);
  PTC_KERNEL("k_cnt_scatter", s, k_cnt_scatter, L.T, kCntThreads, sizeof(ScatterSmem), a);
  PTC_KERNEL("k_cnt_bucket", s, k_cnt_bucket, L.buckets, 1024, sizeof(uint32_t) * kCntBucket, a);
  PTC_KERNEL("k_cnt_out", s, k_cnt_out, ceil_div_u32(n, 2048), 256, 0, a);
  // M and the positions found, beside the status
  uint64_t* hm = host_stage()->out;
  if (copy_to_host_async(hm, L.m, sizeof(uint64_t), s) != PTC_OK) return PTC_ERR_CUDA;
  if (copy_to_host_async(hm + 1, L.found, sizeof(uint32_t), s) != PTC_OK) return PTC_ERR_CUDA;
  DevStatus h;
  const ptc_status rc = end_call(L.st, s, &h);
  *counted = rc != PTC_OK || hm[0] == *reinterpret_cast<const uint32_t*>(hm + 1);
  return rc;
}

}  // namespace ptc
