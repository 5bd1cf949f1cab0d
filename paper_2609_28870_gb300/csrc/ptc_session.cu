// Session-level LRU eviction at every capacity of a grid (Sec. 5.3: block-
// level vs session-level eviction).  Session-level eviction is not a stack
// algorithm (a cache of C + 1 blocks can hold a session that a cache of C
// blocks dropped whole), so each capacity is its own replay: one CTA per
// capacity walks the trace in order.
//
// Readings: a block belongs to the session whose request brought it in,
// until evicted (hits by other sessions do not move it); sessions are ordered
// by their latest request, touched when it arrives; while more than C blocks
// are resident the least recently touched other session loses all its
// blocks; a session that alone holds more than C keeps only the block just
// brought in.  Blocks count with the prefix rule (Sec. 2.2).
//
// State per capacity, all O(1) per step:
//   owner[id]  (session << 32 | epoch) of the session that brought block id
//              in, all ones if never; the block is resident iff that epoch is
//              still its session's current one;
//   epoch[s]   bumped when session s is evicted, which drops all its blocks
//              at once; count[s] its resident blocks;
//   last[s]    its latest request; the requests themselves are the recency
//              queue: the next victim is the oldest request r at the front
//              that is still its session's latest and whose session holds
//              blocks (a passed entry never becomes valid again, so the front
//              only moves forward).
// The replay of one capacity is a serial chain, so what bounds it is the
// latency of a step.  A step settles a window of up to kSesWin accesses of one
// request: each of the replaying warps takes 32 of them (owner, epoch, one
// ballot), a barrier counts the misses, the ballots are exchanged through shared
// memory where there are some, and every warp draws the same conclusions from
// them, so that the replay's state needs no other exchange.  All misses that fit
// settle together; a miss that takes the cache past C evicts (the queue is
// searched 32 requests at a time) and the accesses after it are tested again
// from the owners in registers, since an eviction can drop a later block of the
// window.  Once the current session is alone and above C, every later block of
// the window misses, and they settle in closed form.  Eight other warps read
// ahead: the ids of the next 4,096 accesses into shared memory, and the owner
// words of those ids into L1, so that the owner reads hit L1 (the replayers'
// stores go through the same L1) instead of waiting for L2 or DRAM: the owner
// table takes 8 bytes per block and capacity.  Epochs, counts and latest
// requests sit in shared memory when there are at most kSesSmemSessions sessions.
//
// Ids of prefix chains rise strictly within a request (a prefix first occurs
// no later than its extensions), so no window holds a block twice.  Whether
// the given ids do is checked once for all capacities (k_ses_check); if they
// do not, every window is settled 32 accesses at a time, a second copy of a
// block after the first.
//
// Measured on the 9.3M-access chat trace, 64 capacities: 486 ms with one warp
// per capacity, 32 accesses a step and owners read from DRAM as they came; 116
// ms with 128 accesses a step and the ids read ahead; 55 ms with the epochs read
// together and the check for repeats made once; 41 ms with 16 warps and one
// barrier per eviction (43.9 without the owners read ahead); 36.6 ms with windows
// that start where the last one or its request ended (37.3 with two accesses per
// lane, 1,024 to a window).  The smallest capacities take longest: they evict in
// every window (36.2 ms for 64 blocks, 18.0 for 1.6M).
#include "ptc_internal.h"

namespace ptc {
namespace {

constexpr uint64_t kNoOwner = ~0ULL;

struct SesCaps {
  uint64_t c[PTC_MAX_CAPACITIES];
};

struct SesArgs {
  const uint32_t* ids;
  const uint64_t* blk_off;
  const uint32_t* ses;
  uint32_t n_req, n_session;
  uint64_t n_distinct;
  uint64_t* owner;  // G slices of n_distinct
  uint32_t *epoch, *count, *last;  // G slices of n_session each
  uint64_t sD, sS;
  uint32_t G;
  uint64_t alpha, beta;
  uint64_t* out;  // hits[G] | saved[G] (lo, hi)
  DevStatus* st;
};

__device__ __forceinline__ void add_mul128(uint64_t& lo, uint64_t& hi, uint64_t a, uint64_t b) {
  const uint64_t plo = a * b, phi = __umul64hi(a, b);
  lo += plo;
  hi += phi + (lo < plo ? 1 : 0);
}

// Request offsets and labels checked once (the replay trusts them
// afterwards), ids too, and whether ids rise strictly within every request
// (*falls is raised where they do not).  One thread per access, the first
// n_req of them per request as well.
__global__ void k_ses_check(const uint64_t* __restrict__ blk_off, uint32_t R, uint64_t n,
                            const uint32_t* __restrict__ ses, uint32_t S, const uint32_t* __restrict__ ids,
                            uint64_t D, uint32_t* falls, DevStatus* st) {
  grid_dep_sync();
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < R) {
    const uint64_t a = blk_off[t], b = blk_off[t + 1];
    if (b < a || b > n || (t == 0 && a != 0) || (t + 1 == R && b != n) || ses[t] >= S) raise_err(st, kErrInvalid);
  }
  if (t < n) {
    const uint32_t id = ids[t];
    if (id >= D) raise_err(st, kErrInvalid);
    if (t > 0 && id <= ids[t - 1] && blk_off[req_search(blk_off, 0, R - 1, t)] != t) *falls = 1;
  }
}

// Session state is kept in shared memory up to this many sessions (12 bytes each
// beside the ring), and above it in global memory, of which L1 serves what is in
// use: 136 ms for 14,000 sessions and 140 for 14,400 (the tiny workload's shape,
// 16 capacities).
constexpr uint32_t kSesSmemSessions = 14336;
constexpr uint32_t kSesReplay = 16;            // warps that replay
constexpr uint32_t kSesWin = 32 * kSesReplay;  // accesses per window, one per lane
constexpr uint32_t kSesAhead = 8;              // warps that read ahead
constexpr uint32_t kSesAheadPer = 16;          // accesses per lane that a batch reads ahead
constexpr uint32_t kSesBatch = kSesAhead * 32 * kSesAheadPer;  // 4,096 accesses
constexpr uint32_t kSesThreads = 32 * (kSesReplay + kSesAhead);

// Ids of the batch being replayed and the two after it, and what the replaying
// warps exchange.
struct SesShared {  // the replay's state, where one warp has moved it on alone
  uint64_t total, hits, depths;
  uint32_t cnt, es;
  bool missed;
};
struct SesRing {
  uint32_t ids[3][kSesBatch];
  uint32_t slots[2][32];  // exchanged ballots
  uint32_t touched[kSesAhead];
  SesShared state;
};

// One capacity's session state, in shared or global memory.  Every replaying
// warp reads it, the first one's lane 0 writes it.
struct SesState {
  uint32_t *ep, *count, *last;
};

// The front of the recency queue, and the sessions of the 32 requests around
// it, one per lane.
struct SesFront {
  uint32_t front = 0, base = kNone, ses = 0;
};

// A barrier of the replaying warps.
__device__ __forceinline__ void replay_sync() { asm volatile("bar.sync 1, %0;" ::"r"(32 * kSesReplay) : "memory"); }

// The least recently touched session before request r that holds blocks, or
// kNone.  Whole warps only.
__device__ __forceinline__ uint32_t ses_victim(const SesArgs& a, const SesState& S, uint32_t lane, uint32_t r,
                                               SesFront& q) {
  while (q.front < r) {
    if ((q.front & ~31u) != q.base) {
      q.base = q.front & ~31u;
      q.ses = q.base + lane < a.n_req ? a.ses[q.base + lane] : 0u;
    }
    const uint32_t f = q.base + lane;
    const bool ok =
        f >= q.front && f < r && in_bounds(a.st, q.ses, a.n_session) && S.last[q.ses] == f && S.count[q.ses] > 0;
    const uint32_t m = __ballot_sync(kFull, ok);
    if (m) {
      const uint32_t b = __ffs(m) - 1;
      q.front = q.base + b + 1;
      return __shfl_sync(kFull, q.ses, b);
    }
    q.front = r - q.base > 32 ? q.base + 32 : r;
  }
  return kNone;
}

// Whether owner word `o` names a resident block, where sessions v and w are
// known to have been evicted.
__device__ __forceinline__ bool ses_resident(const SesArgs& a, const SesState& S, uint64_t o, uint32_t v = kNone,
                                             uint32_t w = kNone) {
  const uint32_t t = o == kNoOwner ? 0u : (uint32_t)(o >> 32);
  const uint32_t ep = in_bounds(a.st, t, a.n_session) ? S.ep[t] : 0u;
  return o != kNoOwner && ep == (uint32_t)o && t != v && t != w;
}

// The misses of a window: every warp stores its ballot, and the barrier itself
// counts them.
__device__ __forceinline__ uint32_t ses_count(bool miss, uint32_t* slots, uint32_t warp, uint32_t lane) {
  const uint32_t mine = __ballot_sync(kFull, miss);
  if (lane == 0) slots[warp] = mine;
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.popc.aligned.u32 %0, 1, %2, p;\n\t}"
      : "=r"(all)
      : "r"((uint32_t)miss), "r"(32 * kSesReplay)
      : "memory");
  return all;
}
// Lane w < kSesReplay holds warp w's ballot and the misses of the warps before.
struct SesMisses {
  uint32_t mask, before;
};
__device__ __forceinline__ SesMisses ses_misses(const uint32_t* slots, uint32_t lane) {
  SesMisses m;
  m.mask = lane < kSesReplay ? slots[lane] : 0u;
  const uint32_t c = __popc(m.mask);
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < (int)kSesReplay; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  m.before = x - c;
  return m;
}

template <bool SMEM>
__global__ void __launch_bounds__(kSesThreads, 1) k_ses_sim(SesArgs a, SesCaps caps, uint32_t n,
                                                         const uint32_t* falls) {
  extern __shared__ uint32_t s_dyn[];
  SesRing& ring = *reinterpret_cast<SesRing*>(s_dyn);
  grid_dep_sync();
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t g = blockIdx.x;
  if (g >= a.G) return;
  // malformed offsets, labels or ids: nothing to replay
  if (__syncthreads_or(threadIdx.x == 0 && ld_relaxed_u32(&a.st->err) != 0)) return;
  uint64_t* owner = a.owner + g * a.sD;
  SesState S;
  if (SMEM) {
    S.ep = s_dyn + sizeof(SesRing) / 4;
    S.count = S.ep + a.n_session;
    S.last = S.count + a.n_session;
    for (uint32_t t = threadIdx.x; t < a.n_session; t += kSesThreads) {
      S.ep[t] = 0;
      S.count[t] = 0;
      S.last[t] = kNone;
    }
  } else {  // cleared by the caller
    S.ep = a.epoch + g * a.sS;
    S.count = a.count + g * a.sS;
    S.last = a.last + g * a.sS;
  }
  // The read-ahead warps' share of a batch: the owner words of batch t_owner
  // into L1 and the ids of batch t_ids into the ring, all loads in flight
  // together and once per batch: L1 answers in order, so the replayer's hits
  // wait while any of these misses is outstanding.
  auto read_ahead = [&](uint32_t t_owner, uint32_t t_ids) {
    const uint32_t k0 = (warp - kSesReplay) * 32 * kSesAheadPer + lane;
    const uint64_t owners = (uint64_t)t_owner * kSesBatch, next = (uint64_t)t_ids * kSesBatch;
    uint32_t id[kSesAheadPer], touched = 0;
#pragma unroll
    for (uint32_t u = 0; u < kSesAheadPer; ++u) {
      const uint32_t k = k0 + 32 * u;
      id[u] = next + k < n ? __ldg(&a.ids[next + k]) : 0u;
    }
    if (t_owner != kNone) {
#pragma unroll
      for (uint32_t u = 0; u < kSesAheadPer; ++u) {
        const uint32_t k = k0 + 32 * u;
        if (owners + k < n) touched ^= *reinterpret_cast<const uint32_t*>(owner + ring.ids[t_owner % 3][k]);
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < kSesAheadPer; ++u) ring.ids[t_ids % 3][k0 + 32 * u] = id[u];
    // nobody reads it: without a use the loads that bring the words into L1
    // would be removed
    ring.touched[warp - kSesReplay] = touched;
  };
  const uint64_t C = caps.c[g];
  const uint32_t per = C < kSesWin ? (uint32_t)C : 2 * kSesWin;  // misses between two resets of a lone session
  const uint32_t per_inv = (1u << 20) / per + 1;  // k / per = k per_inv >> 20 for k < kSesWin, per <= 2 kSesWin
  const bool repeats = __ldg(falls) != 0;
  uint64_t total = 0;
  uint64_t hits = 0, depths = 0;  // counted hits and their depths
  SesFront queue;
  // the current request; 32 requests' sessions and ends at a time, one per lane.
  // Every replaying warp keeps all of this.
  uint32_t r = kNone, s = kNone, b = 0, e = 0, es = 0, cnt = 0, q_s = 0, q_e = 0;
  uint32_t turn = 0;  // which of the two sets of exchange slots is next
  const bool writer = threadIdx.x == 0;
  bool missed = false;
  const uint32_t batches = (uint32_t)(((uint64_t)n + kSesBatch - 1) / kSesBatch);
  const bool ahead = warp >= kSesReplay;
  if (ahead) read_ahead(kNone, 0);
  __syncthreads();
  if (ahead) read_ahead(0, 1);
  __syncthreads();
  for (uint32_t t = 0; t < batches; ++t) {
    if (ahead) {
      if (t + 1 < batches) read_ahead(t + 1, t + 2);
      __syncthreads();
      continue;
    }
    const uint32_t* ids = ring.ids[t % 3];
    const uint64_t t0 = (uint64_t)t * kSesBatch;
    const uint32_t size = n - t0 < kSesBatch ? (uint32_t)(n - t0) : kSesBatch;
    uint32_t at = 0;  // accesses of this batch settled
    // The window in registers: this lane's id and owner word.  The next window's
    // are read while this one's misses are counted, the owners again after a step
    // that stored some.
    uint32_t next_id = 0;
    uint64_t next_o = kNoOwner;
    bool ready = false, stale = false;
    auto read_id = [&](uint32_t k) { return ids[k < size ? k : size - 1]; };
    while (at < size) {
      if (t0 + at >= e) {  // the next request with accesses (those without only touch their sessions)
        uint32_t next_s = s;
        do {
          ++r;
          if (r >= a.n_req) break;  // cannot happen: the offsets were checked
          if ((r & 31) == 0) {
            q_s = r + lane < a.n_req ? a.ses[r + lane] : 0u;
            q_e = r + lane < a.n_req ? (uint32_t)a.blk_off[r + lane + 1] : 0u;
          }
          next_s = __shfl_sync(kFull, q_s, r & 31);
          b = e;
          e = __shfl_sync(kFull, q_e, r & 31);
          if (writer) S.last[next_s] = r;
        } while (t0 + at >= e);
        // the new session's count was stored, and every epoch, before the last
        // window's barrier
        if (next_s != s) {
          if (writer && s != kNone) S.count[s] = cnt;
          s = next_s;
          es = S.ep[s];
          cnt = S.count[s];
        }
        missed = false;
      }
      if (t0 + at >= e) break;
      const uint32_t w0 = at;  // the window: up to kSesWin accesses of the request from here
      uint32_t hi = size - w0 < kSesWin ? size - w0 : kSesWin;
      if (e - (t0 + w0) < hi) hi = (uint32_t)(e - (t0 + w0));
      const uint64_t depth = t0 + at - b;
      at = w0 + hi;
      if (repeats) {
        // ---- a block may come twice: 32 accesses at a time, by the first warp
        replay_sync();  // the request's state is written
        if (warp == 0) {
          uint64_t d0 = depth;
          for (uint32_t c = 0; c < hi; c += 32) {
            const uint32_t k = c + lane;
            const uint32_t x = read_id(w0 + k);
            uint32_t pending = __ballot_sync(kFull, k < hi);
            while (pending) {
              const bool mine = (pending >> lane) & 1u;
              const bool res = ses_resident(a, S, mine ? owner[x] : kNoOwner);
              uint32_t same = 0;
              if (mine) same = __match_any_sync(pending, x);
              const uint32_t later_copy = __ballot_sync(kFull, mine && (same & lanemask_lt()) != 0);
              const uint32_t ms = __ballot_sync(kFull, mine && !res);
              const uint64_t room = C - total;
              uint32_t over = 32;  // the first miss that would push the cache past C
              if ((uint64_t)__popc(ms) > room) {
                uint32_t m = ms;
                for (uint64_t q = 0; q < room; ++q) m &= m - 1u;
                over = (uint32_t)(__ffs(m) - 1);
              }
              const uint32_t rep = later_copy ? (uint32_t)(__ffs(later_copy) - 1) : 32u;
              const uint32_t stop = over < rep ? over : rep;
              const uint32_t part = pending & (stop == 32 ? kFull : ((1u << stop) - 1u));
              const uint32_t pm = ms & part;
              __syncwarp();
              if ((pm >> lane) & 1u) owner[x] = ((uint64_t)s << 32) | es;
              total += __popc(pm);
              cnt += __popc(pm);
              if (!missed && part) {
                const uint32_t f0 = __ffs(part) - 1;
                const uint32_t f = (pm ? (uint32_t)(__ffs(pm) - 1) : 32u - __clz(part)) - f0;
                hits += f;
                depths += (uint64_t)f * d0 + (uint64_t)f * (f ? f - 1 : 0) / 2;
                missed = pm != 0;
              }
              d0 += __popc(part);
              pending &= ~part;
              __syncwarp();
              if (stop == 32 || stop == rep) continue;  // done, or a repeated block: test it again
              const uint32_t y = __shfl_sync(kFull, x, stop);
              // one block too many: the least recently touched other session
              // goes whole, or, with none left, this one but for block y
              const uint32_t v = ses_victim(a, S, lane, r, queue);
              if (v == kNone) {
                es += 1;
                cnt = 1;
                total = 1;
              } else {
                cnt += 1;
                total = C + 1 - S.count[v];
              }
              __syncwarp();
              if (writer) {
                owner[y] = ((uint64_t)s << 32) | es;
                if (v == kNone) {
                  S.ep[s] = es;
                } else {
                  S.ep[v] += 1u;
                  S.count[v] = 0;
                }
              }
              __syncwarp();
              missed = true;
              d0 += 1;
              pending &= ~(1u << stop);
            }
          }
          if (writer) ring.state = SesShared{total, hits, depths, cnt, es, missed};
        }
        replay_sync();
        total = ring.state.total;
        hits = ring.state.hits;
        depths = ring.state.depths;
        cnt = ring.state.cnt;
        es = ring.state.es;
        missed = ring.state.missed;
        continue;
      }
      const uint32_t k = 32 * warp + lane;
      const bool valid = k < hi;
      const uint32_t id = ready ? next_id : read_id(w0 + k);
      const uint64_t o = ready && !stale ? next_o : w0 + k < size ? owner[id] : kNoOwner;
      bool miss = valid && !ses_resident(a, S, o);
      ready = at < size;
      if (ready) {
        next_id = read_id(at + k);
        next_o = at + k < size ? owner[next_id] : kNoOwner;
      }
      uint32_t all = ses_count(miss, ring.slots[turn ^= 1], warp, lane);
      stale = all != 0;
      if (all == 0) {
        if (!missed) {
          const uint32_t f = hi;
          hits += f;
          depths += (uint64_t)f * depth + (uint64_t)f * (f - 1) / 2;
        }
        continue;
      }
      if (!missed) {  // the hits before the first miss
        const uint32_t mask = lane < kSesReplay ? ring.slots[turn][lane] : 0u;
        const uint32_t fw = __ffs(__ballot_sync(kFull, mask != 0)) - 1;
        const uint32_t f = 32 * fw + __ffs(__shfl_sync(kFull, mask, fw)) - 1;
        hits += f;
        depths += (uint64_t)f * depth + (uint64_t)f * (f ? f - 1 : 0) / 2;
        missed = true;
      }
      const uint64_t stamp = ((uint64_t)s << 32) | es;
      uint32_t v = kNone;
      while (total + all > C) {
        // the misses before the one that overflows (the room-th, from 0)
        // settle, and so does that one before it evicts
        const uint32_t room = (uint32_t)(C - total);
        const SesMisses m = ses_misses(ring.slots[turn], lane);
        const uint32_t xw =
            __ffs(__ballot_sync(kFull, m.before <= room && m.before + __popc(m.mask) > room)) - 1;
        const uint32_t x_mask = __shfl_sync(kFull, m.mask, xw), x_before = __shfl_sync(kFull, m.before, xw);
        const uint32_t x_lane =
            __ffs(__ballot_sync(kFull, ((x_mask >> lane) & 1u) && x_before + __popc(x_mask & lanemask_lt()) == room)) -
            1;
        const uint32_t x_at = 32 * xw + x_lane;
        const uint32_t v_last = v;
        v = ses_victim(a, S, lane, r, queue);
        if (v == kNone) {
          // session s alone is above C: it keeps the block just brought in, each
          // later one misses, and every C-th of them empties the session again
          if (miss && k < x_at) owner[id] = stamp;
          es += 1;
          const uint32_t rest = hi - 1 - x_at, resets = rest * per_inv >> 20;
          if (k >= x_at && k < hi) owner[id] = ((uint64_t)s << 32) | (es + ((k - x_at) * per_inv >> 20));
          es += resets;
          total = 1 + rest - resets * per;
          cnt = (uint32_t)total;
          all = 0;
          if (writer) S.ep[s] = es;
          break;
        }
        // the least recently touched other session goes whole.  One barrier
        // has to do: the others may still read v's state, so it changes after
        // the barrier, and until the one after that they know v by name.
        if (miss && k <= x_at) owner[id] = stamp;
        cnt += room + 1;
        total = C + 1 - S.count[v];
        miss = valid && k > x_at && !ses_resident(a, S, o, v, v_last);
        all = ses_count(miss, ring.slots[turn ^= 1], warp, lane);
        if (writer) {
          S.ep[v] += 1u;
          S.count[v] = 0;
        }
      }
      if (all) {
        if (miss) owner[id] = stamp;
        total += all;
        cnt += all;
      }
      replay_sync();  // before the next window reads what this one stored
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    uint64_t lo = 0, hi = 0;  // depths fits 64 bits: fewer than 2^32 hits at depths below 2^32
    add_mul128(lo, hi, a.alpha, hits);
    add_mul128(lo, hi, a.beta, depths);
    a.out[g] = hits;
    a.out[a.G + 2 * g] = lo;
    a.out[a.G + 2 * g + 1] = hi;
  }
}

struct SesLayout {
  DevStatus* st;
  uint32_t* falls;  // zeroed with the status block
  uint64_t* owner;
  uint32_t *epoch, *count, *last;
  uint64_t sD, sS;
  uint64_t* out;
  size_t zero_bytes;
  size_t total;
};

SesLayout ses_layout(void* ws, uint64_t n_distinct, uint32_t n_session, uint32_t n_cap) {
  SesLayout L;
  Carver cv(ws);
  const uint64_t G = n_cap ? n_cap : 1;
  L.sD = n_distinct ? n_distinct : 1;
  L.sS = n_session ? n_session : 1;
  L.st = cv.take<DevStatus>(1);
  L.falls = cv.take<uint32_t>(1);
  L.zero_bytes = cv.off;
  L.owner = cv.take<uint64_t>(L.sD * G);
  L.epoch = cv.take<uint32_t>(2 * L.sS * G);  // epochs, then counts: cleared together
  L.count = L.epoch + L.sS * G;
  L.last = cv.take<uint32_t>(L.sS * G);
  L.out = cv.take<uint64_t>(3 * G);
  L.total = cv.bytes();
  return L;
}

}  // namespace
}  // namespace ptc

using namespace ptc;

extern "C" size_t ptc_session_lru_curves_workspace_bytes(uint64_t n_distinct, uint32_t n_session, uint32_t n_cap) {
  return ses_layout(nullptr, n_distinct, n_session, n_cap).total;
}

extern "C" ptc_status ptc_session_lru_curves(const uint32_t* ids, uint64_t n, uint64_t n_distinct,
                                             const uint64_t* req_blk_off, const uint32_t* req_session,
                                             uint32_t n_req, uint32_t n_session, uint32_t block_size,
                                             const ptc_cost_model* cm, const uint64_t* cap_host, uint32_t n_cap,
                                             uint64_t* hits_host_out, ptc_u128* saved_host_out, void* ws,
                                             size_t ws_bytes, void* stream) {
  if (n >= (uint64_t)kNone || n_distinct > n) return PTC_ERR_INVALID_ARG;
  if (!cm || !cap_host || !hits_host_out || !saved_host_out) return PTC_ERR_INVALID_ARG;
  if (n_cap < 1 || n_cap > PTC_MAX_CAPACITIES) return PTC_ERR_INVALID_ARG;
  if (block_size < 1 || block_size > PTC_MAX_BLOCK_SIZE) return PTC_ERR_INVALID_ARG;
  if (n > 0 && (!ids || !req_blk_off || !req_session || n_req == 0 || n_session == 0 || n_distinct == 0))
    return PTC_ERR_INVALID_ARG;
  for (uint32_t g = 0; g < n_cap; ++g)
    if (cap_host[g] < 1 || (g && cap_host[g] <= cap_host[g - 1])) return PTC_ERR_INVALID_ARG;
  uint64_t alpha = 0, beta = 0;
  const ptc_status crc = cost_coeffs(cm, block_size, &alpha, &beta);
  if (crc != PTC_OK) return crc;
  if (n == 0) {
    for (uint32_t g = 0; g < n_cap; ++g) {
      hits_host_out[g] = 0;
      saved_host_out[g] = ptc_u128{0, 0};
    }
    return PTC_OK;
  }
  if (!ws_ok(ws, ws_bytes, ses_layout(nullptr, n_distinct, n_session, n_cap).total)) return PTC_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  const SesLayout L = ses_layout(ws, n_distinct, n_session, n_cap);
  const FillRange zf[4] = {{ws, L.zero_bytes, 0u},
                           {L.owner, sizeof(uint64_t) * L.sD * n_cap, ~0u},
                           {L.epoch, sizeof(uint32_t) * L.sS * n_cap * 2, 0u},  // epoch and count
                           {L.last, sizeof(uint32_t) * L.sS * n_cap, ~0u}};
  if (fill_many_async(zf, 4, s) != PTC_OK) return PTC_ERR_CUDA;
  PTC_KERNEL("k_ses_check", s, k_ses_check, ceil_div_u32(n > n_req ? n : n_req, 256), 256, 0, req_blk_off, n_req, n,
             req_session, n_session, ids, n_distinct, L.falls, L.st);
  SesArgs a;
  a.ids = ids;
  a.blk_off = req_blk_off;
  a.ses = req_session;
  a.n_req = n_req;
  a.n_session = n_session;
  a.n_distinct = n_distinct;
  a.owner = L.owner;
  a.epoch = L.epoch;
  a.count = L.count;
  a.last = L.last;
  a.sD = L.sD;
  a.sS = L.sS;
  a.G = n_cap;
  a.alpha = alpha;
  a.beta = beta;
  a.out = L.out;
  a.st = L.st;
  SesCaps caps;
  for (uint32_t g = 0; g < n_cap; ++g) caps.c[g] = cap_host[g];
  if (n_session <= kSesSmemSessions) {
    const size_t smem = sizeof(SesRing) + 3 * sizeof(uint32_t) * n_session;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(k_ses_sim<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(SesRing) + 3 * sizeof(uint32_t) * kSesSmemSessions)) != cudaSuccess)
      return PTC_ERR_CUDA;
    if (n_cap <= (uint32_t)num_sms())
      PTC_LAUNCH("k_ses_sim", s,
                 launch_l1(k_ses_sim<true>, n_cap, kSesThreads, smem, s, a, caps, (uint32_t)n, L.falls));
    else
      PTC_KERNEL("k_ses_sim", s, k_ses_sim<true>, n_cap, kSesThreads, smem, a, caps, (uint32_t)n, L.falls);
  } else {
    static_assert(sizeof(SesRing) > 48 * 1024, "the ids read ahead alone need more than a kernel has by default");
    if (cudaFuncSetAttribute(k_ses_sim<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SesRing)) !=
        cudaSuccess)
      return PTC_ERR_CUDA;
    PTC_KERNEL("k_ses_sim", s, k_ses_sim<false>, n_cap, kSesThreads, sizeof(SesRing), a, caps, (uint32_t)n, L.falls);
  }
  HostStage* hs = host_stage();
  if (copy_to_host_async(hs->out, L.out, sizeof(uint64_t) * 3 * n_cap, s) != PTC_OK) return PTC_ERR_CUDA;
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
