// Belady's offline optimum at every capacity of a grid at once (Sec. 3.2: the
// offline ceiling every eviction policy is compared with; App. A-B).
//
// Belady's MIN brings every accessed block in and, when the cache then holds
// more than C blocks, evicts the resident block (not the one just brought
// in) whose next access is farthest.  Its hits are reuses (prev[i], i) kept
// resident, and they are exactly the set this interval greedy picks: take
// the reuses in order of their end i; a cache of C blocks holds the block
// being accessed plus C - 1 kept blocks, so think of C - 1 tracks, each free
// from the last position it is busy at; reuse (p, i) is busy at p+1 .. i-1,
// hits iff some track is free by p, and then takes the track freed latest
// among those (best fit), which is free again from i - 1.  A reuse with
// p = i - 1 is busy nowhere and always hits.  (By end time with best fit,
// the greedy keeps the largest set of reuses with at most C - 1 of them busy
// at any access time -- Carlisle and Lloyd 1995 -- and that set is MIN's;
// the oracle's direct MIN simulation is the check.)
//
// Runs.  Accesses i .. i+L-1 whose previous accesses are p .. p+L-1 (a
// request re-reading a context) form a run.  With gap = i - p >= L, step k of
// a run takes the track freed at p + k if there is one (the latest free time
// <= p + k, since the tracks freed in [p, p + k) went to the earlier steps),
// else the latest free time below p, else a never-used track, else it
// misses; its track is then free from i - 1 + k.  So a run needs the free
// bits of [p, p + L), its number of other steps, that many of the latest free
// times below p, and the new free times of its hits.  If p + L = i, step 0's
// new free time i - 1 is the one step L - 1 looks for, handled on its own.  A
// run with gap < L is cut into pieces of length gap, which meet that case.
//
// One warp simulates one capacity.  The free times are a bitmap over access
// positions with three summary levels (a bit per word that may be nonzero,
// cleared when a search finds the word empty) and a lower bound on the
// smallest free time, so a run with nothing free below p learns it at once.
// Runs go in order, up to 1,024 positions at a time: lane l holds word l of
// the 32 that start with p's, and word l of the 32 below them, so every update
// is a plain store of whole words by one lane.
// What bounds the replay is the latency of one run's chain of reads and
// shuffles, hence: the summaries sit in shared memory (a bit per 32 accesses:
// up to about 50M accesses), and the bitmap's last word, which the next run
// extends, stays in a register.  Hits count with the prefix rule (Sec. 2.2): a
// request's accesses before its first miss.
//
// Measured on the 9.3M-access chat trace, 64 capacities: 180 ms with the
// summaries in L2, every update an atomic and one lane searching; 43.7 ms with
// exact summaries in shared memory; 29 ms so (about 260 instructions a run at
// 5.8 cycles each: instruction latency is what is left, as three more warps
// that read the next runs' bitmap words into L1 changed nothing).
#include "ptc_internal.h"

namespace ptc {
namespace {

constexpr uint32_t kBelThreads = 32;  // one warp per capacity
constexpr size_t kBelSmemMax = 200 * 1024;  // summaries in shared memory up to this size

__device__ __forceinline__ uint32_t hi_bit(uint32_t v) { return 31u - __clz(v); }
__device__ __forceinline__ uint32_t mask_le(uint32_t b) { return b == 31 ? kFull : ((2u << b) - 1u); }
__device__ __forceinline__ uint32_t mask_lt(uint32_t b) { return b == 0 ? 0u : (kFull >> (32 - b)); }
// Exclusive prefix over the lanes of c <= 32 (six ballots, whose latencies
// overlap, where a shuffle scan is a chain of five); *total gets the sum.
__device__ __forceinline__ uint32_t lanes_excl(uint32_t c, uint32_t* total) {
  const uint32_t lt = lanemask_lt();
  uint32_t x = 0, t = 0;
#pragma unroll
  for (int b = 0; b < 6; ++b) {
    const uint32_t m = __ballot_sync(kFull, (c >> b) & 1u);
    x += __popc(m & lt) << b;
    t += __popc(m) << b;
  }
  *total = t;
  return x;
}
// The j highest set bits of v, the same v and j in every lane.
__device__ __forceinline__ uint32_t top_bits(uint32_t v, uint32_t j, uint32_t lane) {
  return __ballot_sync(kFull, ((v >> lane) & 1u) && __popc(v >> lane) <= j);
}
// The j lowest set bits of v, the same v and j in every lane.
__device__ __forceinline__ uint32_t low_bits(uint32_t v, uint32_t j, uint32_t lane) {
  return __ballot_sync(kFull, ((v >> lane) & 1u) && __popc(v & mask_le(lane)) <= j);
}

// Request starts: one bit per access in `heads` and `rs`; offsets checked.
__global__ void k_bel_reqs(const uint64_t* __restrict__ blk_off, uint32_t R, uint64_t n, uint32_t* __restrict__ heads,
                           uint32_t* __restrict__ rs, DevStatus* st) {
  grid_dep_sync();
  const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  const uint64_t a = blk_off[r], b = blk_off[r + 1];
  if (b < a || b > n || (r == 0 && a != 0) || (r + 1 == R && b != n)) {
    raise_err(st, kErrInvalid);
    return;
  }
  if (b > a) {
    atomicOr(&heads[a >> 5], 1u << (a & 31));
    atomicOr(&rs[a >> 5], 1u << (a & 31));
  }
}

// Run heads from prev: an access starts a run unless it and the one before
// are both cold, or both reuses with previous accesses one apart.
__global__ void k_bel_heads(const uint32_t* __restrict__ prev, uint32_t n, uint32_t* __restrict__ heads,
                            DevStatus* st) {
  grid_dep_sync();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  bool head = false;
  if (i < n) {
    const uint32_t p = prev[i], q = i ? prev[i - 1] : kNone;
    if (p != kNone && p >= i) raise_err(st, kErrInvalid);  // a previous access lies before
    head = i == 0 || (p == kNone) != (q == kNone) || (p != kNone && p != q + 1);
  }
  const uint32_t b = __ballot_sync(kFull, head);
  if ((threadIdx.x & 31) == 0 && b && i < n) atomicOr(&heads[i >> 5], b);
}

// Run records at the heads' ranks: first access, its previous access (kNone
// for a run of cold accesses), whether it opens a request; rec_start[runs] = n.
__global__ void k_bel_records(const uint32_t* __restrict__ prev, uint32_t n, const uint32_t* __restrict__ heads,
                              const uint32_t* __restrict__ rs, const uint32_t* __restrict__ wpre,
                              const uint64_t* __restrict__ nruns, uint32_t* __restrict__ rec_start,
                              uint32_t* __restrict__ rec_p, uint8_t* __restrict__ rec_rs) {
  grid_dep_sync();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) rec_start[*nruns] = n;
  if (i >= n) return;
  const uint32_t w = heads[i >> 5], bit = 1u << (i & 31);
  if (!(w & bit)) return;
  const uint32_t r = wpre[i >> 5] + __popc(w & (bit - 1u));
  rec_start[r] = i;
  rec_p[r] = prev[i];
  rec_rs[r] = (rs[i >> 5] & bit) ? 1 : 0;
}

struct BelCaps {
  uint64_t c[PTC_MAX_CAPACITIES];
};

struct BelArgs {
  const uint32_t* rec_start;
  const uint32_t* rec_p;
  const uint8_t* rec_rs;
  const uint64_t* nruns;
  uint32_t *lv0, *sum;        // free-time bitmap and its summaries, one slice per capacity
  uint32_t s0, s1, s2, s3;    // words per slice and level (sum: s1 + s2 + s3)
  uint32_t G;
  uint64_t alpha, beta;
  uint64_t* out;  // hits[G] | saved[G] (lo, hi) | raw hits[G]
  const DevStatus* st;
};

// One capacity's free-time bitmap: level 0 one bit per access position,
// level k + 1 one bit per word of level k that may be nonzero (a nonzero word
// always has its bit).  Only one warp uses it, every lane calling each
// function.  `low` is a lower bound on every set position (raised when a
// search finds nothing below a point).
struct FreeBits {
  uint32_t *l0, *l1, *l2, *l3;
  uint32_t low;
  uint32_t words;  // level-0 words of the slice
  const DevStatus* st;

  // Words w0 .. w0 + 31 became nonzero where `m` is set.  They meet two words
  // of level 1, which held old0 and old1 (stale bits may be among them).
  __device__ __forceinline__ void mark(uint32_t w0, uint32_t m, uint32_t old0, uint32_t old1, uint32_t lane) {
    const uint32_t sh = w0 & 31, w1 = w0 >> 5;
    const uint32_t b0 = m << sh, b1 = sh ? m >> (32 - sh) : 0u;
    if (lane == 0) {
      if (b0) l1[w1] = old0 | b0;
      if (b1) l1[w1 + 1] = old1 | b1;
    }
    if ((b0 && !old0) || (b1 && !old1)) {
      if (lane == 0) {
        if (b0) {
          l2[w1 >> 5] |= 1u << (w1 & 31);
          l3[w1 >> 10] |= 1u << ((w1 >> 5) & 31);
        }
        if (b1) {
          l2[(w1 + 1) >> 5] |= 1u << ((w1 + 1) & 31);
          l3[(w1 + 1) >> 10] |= 1u << (((w1 + 1) >> 5) & 31);
        }
      }
    }
    __syncwarp();
  }
  // The highest word of level 1 below word w1 that is nonzero, or kNone;
  // level-2 and level-3 bits of words found empty are cleared on the way.
  __device__ __forceinline__ uint32_t below1(uint32_t w1, uint32_t lane) {
    uint32_t w2 = w1 >> 5, m2 = l2[w2] & mask_lt(w1 & 31);
    while (true) {
      while (m2) {
        const uint32_t b = hi_bit(m2), c = w2 * 32 + b;
        if (l1[c]) return c;
        if (lane == 0) l2[w2] &= ~(1u << b);
        m2 &= ~(1u << b);
        __syncwarp();
      }
      uint32_t w3 = w2 >> 5, m3 = l3[w3] & mask_lt(w2 & 31);
      while (!m3) {
        if (w3 == 0) return kNone;
        m3 = l3[--w3];
      }
      w2 = w3 * 32 + hi_bit(m3);
      m2 = l2[w2];
      __syncwarp();
      if (!m2 && lane == 0) l3[w3] &= ~(1u << (w2 & 31));
      __syncwarp();
    }
  }
  // Clear the `need` highest set bits in the words below word `end`; returns
  // how many there were (fewer if the bitmap runs out).  32 words at a time,
  // lane l the l-th of those under one word of level 1, in falling order.
  __device__ __forceinline__ uint32_t pop_words(uint32_t end, uint32_t need, uint32_t lane) {
    uint32_t got = 0, w1 = end >> 5;
    uint32_t m1 = l1[w1] & mask_lt(end & 31);
    while (true) {
      if (m1) {
        const uint32_t b = 31 - lane, w = w1 * 32 + b;
        const uint32_t v = ((m1 >> b) & 1u) && in_bounds(st, w, words) ? l0[w] : 0u;
        uint32_t sum;
        const uint32_t c = __popc(v), above = lanes_excl(c, &sum);
        const uint32_t want = need - got;
        uint32_t take = above + c <= want ? v : 0u;
        const uint32_t part = __ballot_sync(kFull, above < want && above + c > want);
        if (part) {  // the word that holds the last one wanted
          const uint32_t src = __ffs(part) - 1;
          const uint32_t t = top_bits(__shfl_sync(kFull, v, src), want - __shfl_sync(kFull, above, src), lane);
          if (lane == src) take = t;
        }
        if (take) l0[w] = v & ~take;
        const uint32_t empty = m1 & __brev(__ballot_sync(kFull, v == take));
        if (lane == 0 && empty) l1[w1] &= ~empty;
        __syncwarp();
        if (sum >= want) return need;
        got += sum;
      }
      w1 = w1 ? below1(w1, lane) : kNone;
      if (w1 == kNone) return got;
      m1 = l1[w1];
    }
  }
};

__device__ __forceinline__ void add128(uint64_t& lo, uint64_t& hi, uint64_t a_lo, uint64_t a_hi) {
  lo += a_lo;
  hi += a_hi + (lo < a_lo ? 1 : 0);
}
__device__ __forceinline__ void add_mul(uint64_t& lo, uint64_t& hi, uint64_t a, uint64_t b) {
  add128(lo, hi, a * b, __umul64hi(a, b));
}

// One CTA of one warp per capacity.
template <bool SMEM>
__global__ void __launch_bounds__(kBelThreads, 1) k_bel_sim(BelArgs a, BelCaps caps) {
  extern __shared__ uint32_t s_sum[];
  grid_dep_sync();
  const uint32_t lane = threadIdx.x;
  const uint32_t g = blockIdx.x;
  if (g >= a.G) return;
  uint32_t* const l0 = a.lv0 + (uint64_t)g * a.s0;
  uint32_t* const sum = SMEM ? s_sum : a.sum + (uint64_t)g * (a.s1 + a.s2 + a.s3);
  if (SMEM)
    for (uint32_t i = threadIdx.x; i < a.s1 + a.s2 + a.s3; i += kBelThreads) sum[i] = 0;
  FreeBits fb{l0, sum, sum + a.s1, sum + a.s1 + a.s2, 0, a.s0, a.st};
  const uint32_t R = (uint32_t)*a.nruns;
  uint64_t free_inf = caps.c[g] - 1;  // never-used tracks
  uint64_t hits = 0, raw = 0, depths = 0;  // counted hits, all hits, and the counted hits' depths
  uint32_t req_start = 0;
  uint32_t tail_w = 0, tail = 0;  // the highest word that free times were added to, as it stands
  bool missed = false;
  __syncwarp();
  for (uint32_t q0 = 0; q0 < R; q0 += 32) {
    const uint32_t rl = q0 + lane;
    const uint32_t my_s = rl < R ? a.rec_start[rl] : 0u;
    const uint32_t my_e = rl < R ? a.rec_start[rl + 1] : 0u;
    const uint32_t my_p = rl < R ? a.rec_p[rl] : kNone;
    const uint32_t opens = __ballot_sync(kFull, rl < R && a.rec_rs[rl]);  // runs that open a request
    const uint32_t nr = R - q0 < 32 ? R - q0 : 32;
    for (uint32_t t = 0; t < nr; ++t) {
      uint32_t s = __shfl_sync(kFull, my_s, t);
      const uint32_t e = __shfl_sync(kFull, my_e, t);
      uint32_t p = __shfl_sync(kFull, my_p, t);
      if ((opens >> t) & 1u) {
        req_start = s;
        missed = false;
      }
      uint32_t L = e - s;
      if (p == kNone || p >= s) {  // cold accesses: misses, no track (p >= s is malformed, reported)
        missed = true;
        continue;
      }
      if (s - p == 1) {  // every step re-reads the block just accessed: busy nowhere, hits
        raw += L;
        if (!missed) {
          hits += L;
          depths += (uint64_t)L * (s - req_start) + (uint64_t)L * (L - 1) / 2;
        }
        continue;
      }
      while (L > 0) {
        const uint32_t gap = s - p, sp = p & 31;
        uint32_t Lj = L < gap ? L : gap;
        if (Lj > 1024 - sp) Lj = 1024 - sp;  // the 32 words from p's
        // this lane's word of them (positions 32 (w0 + lane) ..) and of the 32 below
        const uint32_t w0 = p >> 5, w = w0 + lane;
        const uint32_t end = sp + Lj;  // past the last step, counted from word w0
        uint32_t valid = lane * 32 >= end ? 0u : end - lane * 32 >= 32 ? kFull : mask_lt(end - lane * 32);
        const bool has = valid != 0 && in_bounds(a.st, w, a.s0);
        const uint32_t word = has ? l0[w] : 0u;
        const uint32_t below = w0 > lane ? l0[w0 - 1 - lane] : 0u;
        // the level-1 words of the 32 words where this chunk's free times go
        const uint32_t v0 = (s - 1) >> 5;
        uint32_t old0 = fb.l1[v0 >> 5], old1 = fb.l1[(v0 >> 5) + 1];
        if (lane == 0) valid &= ~mask_lt(sp);
        const uint32_t Bk = word & valid;
        const bool edge = Lj >= 2 && p + Lj == s;  // the last step: decided by step 0 below
        const uint32_t elane = (end - 1) >> 5, ebit = 1u << ((end - 1) & 31);
        const uint32_t z = Lj - edge - __reduce_add_sync(kFull, __popc(Bk));
        uint32_t left = word & ~valid;  // the free times of [p, p + Lj) are used up
        uint32_t A = valid;        // steps that hit
        uint32_t nh = Lj, f = Lj;  // hits, and hits before the first miss
        if (z) {
          // the other steps take the latest free times below p, then never-used tracks
          uint32_t acc = 0;
          if (p > fb.low) {
            const uint32_t first = __shfl_sync(kFull, word, 0) & mask_lt(sp);  // those in p's own word
            uint32_t sum;
            const uint32_t c = __popc(below), n0 = __popc(first), above = n0 + lanes_excl(c, &sum);
            if (n0 > z) {
              const uint32_t tk = top_bits(first, z, lane);
              if (lane == 0) left &= ~tk;
            } else {
              if (lane == 0) left &= ~first;
              uint32_t take = above + c <= z ? below : 0u;
              const uint32_t part = __ballot_sync(kFull, above < z && above + c > z);
              if (part) {  // the word that holds the last one wanted
                const uint32_t src = __ffs(part) - 1;
                const uint32_t more = z - __shfl_sync(kFull, above, src);
                const uint32_t tk = top_bits(__shfl_sync(kFull, below, src), more, lane);
                if (lane == src) take = tk;
              }
              if (take) l0[w0 - 1 - lane] = below & ~take;
            }
            acc = n0 + sum;
            if (acc >= z) {
              acc = z;
            } else {
              if (w0 > 32) {
                acc += fb.pop_words(w0 - 32, z - acc, lane);
                old0 = fb.l1[v0 >> 5];  // it may have cleared bits there
                old1 = fb.l1[(v0 >> 5) + 1];
              }
              if (acc < z) fb.low = p;  // nothing is left below p, and free times are added above it
            }
          }
          const uint32_t rest = z - acc, inf = rest < free_inf ? rest : (uint32_t)free_inf;
          free_inf -= inf;
          acc += inf;
          if (acc < z) {  // the first acc of them hit
            uint32_t zm = ~Bk & valid, sum;
            if (edge && lane == elane) zm &= ~ebit;
            const uint32_t zc = __popc(zm), zx = lanes_excl(zc, &sum);
            A = (valid & ~zm) | (zx + zc <= acc ? zm : 0u);
            const uint32_t part = __ballot_sync(kFull, zx < acc && zx + zc > acc);
            if (part) {
              const uint32_t src = __ffs(part) - 1;
              const uint32_t tk = low_bits(__shfl_sync(kFull, zm, src), acc - __shfl_sync(kFull, zx, src), lane);
              if (lane == src) A |= tk;
            }
            const bool hit0 = ((__shfl_sync(kFull, Bk, 0) >> sp) & 1u) || acc >= 1;
            if (edge && !hit0 && lane == elane) A &= ~ebit;
            const uint32_t rej = valid & ~A;
            const uint32_t with = __ballot_sync(kFull, rej != 0);
            nh = Lj - __reduce_add_sync(kFull, __popc(rej));
            const uint32_t l_f = __ffs(with) - 1;
            f = 32 * l_f + __ffs(__shfl_sync(kFull, rej, l_f)) - 1 - sp;
          }
        }
        if (has && left != word) l0[w] = left;
        // New free times s - 1 + k of the hits; with p + Lj = s the last step
        // took step 0's.  They lie above every free time so far.
        {
          uint32_t T = A;
          if (edge && lane == 0) T &= ~(1u << sp);
          const uint32_t sq = (s - 1) & 31;
          const uint32_t up = __shfl_up_sync(kFull, T, 1), dn = __shfl_down_sync(kFull, T, 1);
          uint32_t out, past = 0;  // words v0 + lane, and v0 + 32 (lane 31)
          if (sq >= sp) {
            const uint32_t d = sq - sp;
            out = T << d | (d && lane ? up >> (32 - d) : 0u);
            if (d && lane == 31) past = T >> (32 - d);
          } else {
            const uint32_t d = sp - sq;
            out = T >> d | (lane < 31 ? dn << (32 - d) : 0u);
          }
          // what word v0 holds already: the tail's bits, read back if this
          // run's updates may have met that word
          if ((p + Lj - 1) >> 5 >= v0) {
            __syncwarp();  // the words cleared above
            tail_w = v0;
            tail = in_bounds(a.st, v0, a.s0) ? l0[v0] : 0u;
            if (lane == 0 && out) out |= tail;
            __syncwarp();
          } else if (v0 == tail_w && lane == 0 && out) {
            out |= tail;
          }
          if (out && in_bounds(a.st, v0 + lane, a.s0)) l0[v0 + lane] = out;
          if (past && in_bounds(a.st, v0 + 32, a.s0)) l0[v0 + 32] = past;
          const uint32_t set = __ballot_sync(kFull, out != 0);
          fb.mark(v0, set, old0, old1, lane);
          const uint32_t over = __shfl_sync(kFull, past, 31);
          if (over) {
            fb.mark(v0 + 32, 1u, fb.l1[(v0 >> 5) + 1], 0u, lane);
            tail_w = v0 + 32;
            tail = over;
          } else if (set) {
            const uint32_t l_t = hi_bit(set);
            tail_w = v0 + l_t;
            tail = __shfl_sync(kFull, out, l_t);
          }
        }
        raw += nh;
        if (!missed) {
          hits += f;
          depths += (uint64_t)f * (s - req_start) + (uint64_t)f * (f ? f - 1 : 0) / 2;
          if (f < Lj) missed = true;
        }
        s += Lj;
        p += Lj;
        L -= Lj;
      }
    }
  }
  uint64_t sv_lo = 0, sv_hi = 0;  // depths fits 64 bits: fewer than 2^32 hits at depths below 2^32
  add_mul(sv_lo, sv_hi, a.alpha, hits);
  add_mul(sv_lo, sv_hi, a.beta, depths);
  if (threadIdx.x == 0) {
    a.out[g] = hits;
    a.out[a.G + 2 * g] = sv_lo;
    a.out[a.G + 2 * g + 1] = sv_hi;
    a.out[3 * a.G + g] = raw;
  }
}

struct BelLayout {
  DevStatus* st;
  uint32_t* done;
  uint32_t *heads, *rs;  // zeroed with the status block
  uint32_t *wpre, *tcnt, *tpre;
  uint64_t* nruns;
  uint32_t *rec_start, *rec_p;
  uint8_t* rec_rs;
  uint32_t *lv0, *sum;
  uint64_t s0, s1, s2, s3;
  uint64_t* out;
  size_t zero_bytes, bits_bytes;
  uint32_t nwords;
  size_t total;
};

BelLayout bel_layout(void* ws, uint64_t n, uint32_t n_cap) {
  BelLayout L;
  Carver cv(ws);
  const uint64_t nn = n ? n : 1;
  L.nwords = ceil_div_u32(nn, 32);
  L.st = cv.take<DevStatus>(1);
  L.done = cv.take<uint32_t>(64);
  L.heads = cv.take<uint32_t>(L.nwords + 1);
  L.rs = cv.take<uint32_t>(L.nwords + 1);
  L.zero_bytes = cv.off;
  L.wpre = cv.take<uint32_t>(L.nwords + 1);
  L.tcnt = cv.take<uint32_t>(rank_tiles(L.nwords) + 1);
  L.tpre = cv.take<uint32_t>(rank_tiles(L.nwords) + 1);
  L.nruns = cv.take<uint64_t>(1);
  L.rec_start = cv.take<uint32_t>(nn + 1);
  L.rec_p = cv.take<uint32_t>(nn);
  L.rec_rs = cv.take<uint8_t>(nn);
  const uint64_t G = n_cap ? n_cap : 1;
  L.s0 = ((uint64_t)L.nwords + 2 + 31) / 32 * 32;  // whole 128-byte lines
  L.s1 = (L.s0 + 31) / 32 + 1;
  L.s2 = (L.s1 + 31) / 32 + 1;
  L.s3 = (L.s2 + 31) / 32 + 1;
  L.lv0 = cv.take<uint32_t>((L.s0 + L.s1 + L.s2 + L.s3) * G);
  L.sum = L.lv0 + L.s0 * G;
  L.bits_bytes = sizeof(uint32_t) * (L.s0 + L.s1 + L.s2 + L.s3) * G;
  L.out = cv.take<uint64_t>(4 * G);
  L.total = cv.bytes();
  return L;
}

}  // namespace
}  // namespace ptc

using namespace ptc;

extern "C" size_t ptc_belady_curves_workspace_bytes(uint64_t n, uint32_t n_req, uint32_t n_cap) {
  (void)n_req;
  return bel_layout(nullptr, n, n_cap).total;
}

extern "C" ptc_status ptc_belady_curves(const uint32_t* prev, uint64_t n, const uint64_t* req_blk_off,
                                        uint32_t n_req, uint32_t block_size, const ptc_cost_model* cm,
                                        const uint64_t* cap_host, uint32_t n_cap, uint64_t* hits_host_out,
                                        ptc_u128* saved_host_out, uint64_t* raw_hits_host_out, void* ws,
                                        size_t ws_bytes, void* stream) {
  if (n >= (uint64_t)kNone) return PTC_ERR_OVERFLOW;
  if (!cm || !cap_host || !hits_host_out || !saved_host_out) return PTC_ERR_INVALID_ARG;
  if (n_cap < 1 || n_cap > PTC_MAX_CAPACITIES) return PTC_ERR_INVALID_ARG;
  if (block_size < 1 || block_size > PTC_MAX_BLOCK_SIZE) return PTC_ERR_INVALID_ARG;
  if (n > 0 && (!prev || !req_blk_off || n_req == 0)) return PTC_ERR_INVALID_ARG;
  for (uint32_t g = 0; g < n_cap; ++g)
    if (cap_host[g] < 1 || (g && cap_host[g] <= cap_host[g - 1])) return PTC_ERR_INVALID_ARG;
  uint64_t alpha = 0, beta = 0;
  const ptc_status crc = cost_coeffs(cm, block_size, &alpha, &beta);
  if (crc != PTC_OK) return crc;
  if (!ws_ok(ws, ws_bytes, bel_layout(nullptr, n, n_cap).total)) return PTC_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  const BelLayout L = bel_layout(ws, n, n_cap);
  if (n == 0) {
    for (uint32_t g = 0; g < n_cap; ++g) {
      hits_host_out[g] = 0;
      saved_host_out[g] = ptc_u128{0, 0};
      if (raw_hits_host_out) raw_hits_host_out[g] = 0;
    }
    return PTC_OK;
  }
  const FillRange zf[2] = {{ws, L.zero_bytes, 0u}, {L.lv0, L.bits_bytes, 0u}};
  if (fill_many_async(zf, 2, s) != PTC_OK) return PTC_ERR_CUDA;
  const uint32_t n32 = (uint32_t)n;
  PTC_KERNEL("k_bel_reqs", s, k_bel_reqs, ceil_div_u32(n_req, 256), 256, 0, req_blk_off, n_req, n, L.heads, L.rs,
             L.st);
  PTC_KERNEL("k_bel_heads", s, k_bel_heads, ceil_div_u32(n, 256), 256, 0, prev, n32, L.heads, L.st);
  if (bitmap_ranks(L.heads, L.nwords, L.wpre, L.tcnt, L.tpre, L.done, L.nruns, s) != PTC_OK) return PTC_ERR_CUDA;
  PTC_KERNEL("k_bel_records", s, k_bel_records, ceil_div_u32(n, 256), 256, 0, prev, n32, L.heads, L.rs, L.wpre,
             L.nruns, L.rec_start, L.rec_p, L.rec_rs);
  BelArgs a;
  a.rec_start = L.rec_start;
  a.rec_p = L.rec_p;
  a.rec_rs = L.rec_rs;
  a.nruns = L.nruns;
  a.lv0 = L.lv0;
  a.sum = L.sum;
  a.s0 = (uint32_t)L.s0;
  a.s1 = (uint32_t)L.s1;
  a.s2 = (uint32_t)L.s2;
  a.s3 = (uint32_t)L.s3;
  a.G = n_cap;
  a.alpha = alpha;
  a.beta = beta;
  a.out = L.out;
  a.st = L.st;
  BelCaps caps;
  for (uint32_t g = 0; g < n_cap; ++g) caps.c[g] = cap_host[g];
  const size_t sums = sizeof(uint32_t) * (L.s1 + L.s2 + L.s3);
  if (sums <= kBelSmemMax) {
    if (sums > 48 * 1024 && cudaFuncSetAttribute(k_bel_sim<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)kBelSmemMax) != cudaSuccess)
      return PTC_ERR_CUDA;
    if (n_cap <= (uint32_t)num_sms())
      PTC_LAUNCH("k_bel_sim", s, launch_l1(k_bel_sim<true>, n_cap, kBelThreads, sums, s, a, caps));
    else
      PTC_KERNEL("k_bel_sim", s, k_bel_sim<true>, n_cap, kBelThreads, sums, a, caps);
  } else {
    PTC_KERNEL("k_bel_sim", s, k_bel_sim<false>, n_cap, kBelThreads, 0, a, caps);
  }
  HostStage* hs = host_stage();
  if (copy_to_host_async(hs->out, L.out, sizeof(uint64_t) * 3 * n_cap, s) != PTC_OK) return PTC_ERR_CUDA;
  if (raw_hits_host_out &&
      cudaMemcpyAsync(raw_hits_host_out, L.out + 3 * n_cap, sizeof(uint64_t) * n_cap, cudaMemcpyDeviceToHost, s) !=
          cudaSuccess)
    return PTC_ERR_CUDA;
  DevStatus h;
  const ptc_status rc = end_call(L.st, s, &h);
  if (rc != PTC_OK) return rc;
  for (uint32_t g = 0; g < n_cap; ++g) {
    hits_host_out[g] = hs->out[g];
    saved_host_out[g].lo = hs->out[n_cap + 2 * g];
    saved_host_out[g].hi = hs->out[n_cap + 2 * g + 1];
  }
  return PTC_OK;
}
