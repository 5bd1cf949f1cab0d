// Stage a1: chained block keys (paper Sec. 2.2 block identity).
//
// Block k of a request covers tokens [Bk, Bk+B).  Its key is a polynomial of
// the whole prefix over GF(2^61 - 1) at two seeded bases u (one per key word):
//     S_k = sum_{t < B(k+1)} (tok_t + 1) u^(t+1)
// Every coefficient is at least 1, so two different prefixes, of equal or of
// different length, differ as polynomials (Karp-Rabin; a pair collides with
// probability at most length / 2^61 per base).  Written per block:
//     h_j = sum_{i<B} (tok_{Bj+i} + 1) u^(i+1)                 (block-local)
//     S_k = sum_{j<=k} h_j u^(Bj)
// so the chain across a request is a plain segmented sum of g_j = h_j u^(Bj):
// one scan, no sequential chain, and the sum itself is the key.
//
// Kernels
//   k_block_offsets  per-request block counts -> exclusive scan (look-back),
//                    validates offsets, timestamp order and session labels;
//                    CTAs beside those of the scan fill the powers u^(U e),
//                    two levels of 65,536 entries, as far as a request can reach
//   k_hash_units     B a multiple of 16, 12 or 8: a unit of U = 16, 12 or 8
//                    tokens per lane, 32 units at a time, then prefix sums over
//                    the units of a warp's tile, 8, 9 or 11 per lane
//                    (three-limb products where a token reaches 2^27)
//   k_hash_local     any other B: tokens
//                    staged through padded shared memory with 16-byte
//                    loads; each thread hashes 16 tokens (one "sub-chunk")
//                    with 3 x 21-bit limbs of u^1..u^16 held as constant
//                    kernel parameters; sub-chunks of one block combine by
//                    shuffles; the segmented sum runs across the CTA.  Keys
//                    after the tile's first request start are final; the tile
//                    records its aggregate.  No tile depends on another.
//   k_hash_chain     each tile's carry from its predecessors' aggregates
//                    (all already written, so nothing waits), added to the
//                    keys of the tile's leading blocks.
#include "ptc_internal.h"

namespace ptc {
namespace {

constexpr int kOffThreads = 256;  // one request per thread: the grid spreads over many SMs
constexpr int kOffPer = 1;
constexpr int kOffTile = kOffThreads * kOffPer;

constexpr int kHashThreads = 256;
constexpr int kWinTokens = 8192 + 256;
constexpr int kWinWords = kWinTokens + kWinTokens / 16;

constexpr int kEpochOffsets = 1;

// ---------------------------------------------------------------- block scans
// Exclusive sum over a CTA of kOffThreads threads; returns the CTA total in *total.
__device__ __forceinline__ uint64_t cta_exclusive_sum(uint64_t v, uint64_t* total) {
  __shared__ uint64_t s_w[kOffThreads / 32];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint64_t y = __shfl_up_sync(kFull, x, d);
    if (lane >= (uint32_t)d) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    uint64_t t = lane < kOffThreads / 32 ? s_w[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      uint64_t y = __shfl_up_sync(kFull, t, d);
      if (lane >= (uint32_t)d) t += y;
    }
    if (lane < kOffThreads / 32) s_w[lane] = t;  // inclusive over warps
  }
  __syncthreads();
  uint64_t warp_excl = w ? s_w[w - 1] : 0;
  *total = s_w[kOffThreads / 32 - 1];
  return warp_excl + x - v;
}

// ---------------------------------------------------------------- powers
// tables[(b*2 + w) * 65536 + e] for base b in {0,1} and U tokens per unit
// (k_hash_local: a unit is a block)
//   w = 0: u_b^(U e)          w = 1: u_b^(U 65536 e)
// The first n_lo and n_hi entries are filled: as many as the longest request
// that the tokens allow can use.
constexpr int kPowChunk = 8;  // powers per thread: short dependent chains

struct PowArgs {
  uint64_t base[4];
  uint64_t* tables;
  uint32_t n_lo, n_hi;
  uint32_t off_tiles;  // CTAs of the offsets' scan; the others fill powers
};
inline uint32_t pow_chunks(const PowArgs& p) {
  return 2 * (ceil_div_u32(p.n_lo, kPowChunk) + ceil_div_u32(p.n_hi, kPowChunk));
}

__device__ __forceinline__ void fill_powers(const PowArgs& p, uint32_t chunk) {
  const uint32_t c_lo = (p.n_lo + kPowChunk - 1) / kPowChunk, c_hi = (p.n_hi + kPowChunk - 1) / kPowChunk;
  uint32_t t = 0, n = p.n_lo;
  if (chunk >= c_lo + c_hi) {
    t = 2;
    chunk -= c_lo + c_hi;
  }
  if (chunk >= c_lo) {
    ++t;
    chunk -= c_lo;
    n = p.n_hi;
    if (chunk >= c_hi) return;
  }
  const uint64_t base = p.base[t];
  const uint32_t e0 = chunk * kPowChunk;
  uint64_t v = p61_pow(base, e0);
  uint64_t* out = p.tables + (uint64_t)t * 65536 + e0;
  for (uint32_t i = 0; i < (uint32_t)kPowChunk && e0 + i < n; ++i) {
    out[i] = v;
    v = p61_mul(v, base);
  }
}

__global__ void __launch_bounds__(kOffThreads) k_block_offsets(const uint64_t* __restrict__ tok_off,
                                                               const int64_t* __restrict__ ts, uint32_t R,
                                                               uint64_t n_tok, uint32_t B, uint32_t tb,
                                                               uint64_t* __restrict__ blk_off,
                                                               uint32_t* __restrict__ tile_req, uint64_t tile_cap,
                                                               uint64_t* lb, DevStatus* st,
                                                               const uint32_t* __restrict__ ses,
                                                               uint32_t n_session,
                                                               const __grid_constant__ PowArgs pw) {
  grid_dep_sync();
  if (blockIdx.x >= pw.off_tiles) {
    fill_powers(pw, (blockIdx.x - pw.off_tiles) * kOffThreads + threadIdx.x);
    return;
  }
  const uint32_t tile = next_tile(st, kEpochOffsets);
  const uint64_t r0 = (uint64_t)tile * kOffTile + (uint64_t)threadIdx.x * kOffPer;
  uint64_t cnt[kOffPer];
  uint64_t local = 0, kmax = 0;
  uint32_t err = 0;
#pragma unroll
  for (int j = 0; j < kOffPer; ++j) {
    uint64_t r = r0 + j;
    cnt[j] = 0;
    if (r < R) {
      uint64_t a = tok_off[r], b = tok_off[r + 1];
      if (b < a || b > n_tok) {
        err |= kErrInvalid;
      } else {
        cnt[j] = (b - a) / B;
      }
      if (ts != nullptr && r + 1 < R && ts[r + 1] < ts[r]) err |= kErrUnsorted;
      if (ses != nullptr && ses[r] >= n_session) err |= kErrInvalid;
      local += cnt[j];
      kmax = cnt[j] > kmax ? cnt[j] : kmax;
    }
  }
  if (err) raise_err(st, err);
  {  // the longest request: one atomic per warp
    uint64_t m = kmax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t y = __shfl_xor_sync(kFull, m, o);
      m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax((unsigned long long*)&st->value[1], (unsigned long long)m);
  }
  uint64_t total;
  uint64_t excl = cta_exclusive_sum(local, &total);
  const uint64_t base = lookback_sum_cta(lb, tile, total, kEpochOffsets, st);
  uint64_t run = base + excl;
#pragma unroll
  for (int j = 0; j < kOffPer; ++j) {
    uint64_t r = r0 + j;
    if (r < R) {
      blk_off[r] = run;
      // hash tiles whose first block lies in this request
      if (cnt[j]) {
        const uint64_t last = (run + cnt[j] - 1) / tb;
        for (uint64_t t = (run + tb - 1) / tb; t <= last && t < tile_cap; ++t) tile_req[t] = (uint32_t)r;
      }
    }
    run += cnt[j];
    if (r + 1 == R) {
      blk_off[R] = run;
      st->value[0] = run;
      if (run >= (uint64_t)kNone) raise_err(st, kErrOverflow);
    }
  }
}

// Blocks the key kernels may touch: N as the offsets kernel left it, or none
// if its look-back gave up (then the offsets are not a prefix sum and must
// not steer any read; the call reports PTC_ERR_TIMEOUT).
__device__ __forceinline__ uint64_t blocks_live(const DevStatus* st, uint64_t keys_cap) {
  if (ld_relaxed_u32(&st->err) & kErrTimeout) return 0;
  const uint64_t N = st->value[0];
  return N < keys_cap ? N : keys_cap;
}

__device__ __forceinline__ uint64_t pow_at(const uint64_t* __restrict__ lo, const uint64_t* __restrict__ hi,
                                           uint64_t e) {
  uint64_t v = __ldg(&lo[e & 0xFFFF]);
  const uint64_t h = e >> 16;
  if (h) v = p61_mul(v, __ldg(&hi[h & 0xFFFF]));
  return v;
}

// ---------------------------------------------------------------- hash
struct HashConsts {
  uint32_t limb[2][3][16];   // 21-bit limbs of u_b^(j + 1)
  uint32_t limb2[2][2][16];  // the same split 31 + 30 bits (tokens below 2^27)
  uint64_t csum[2][17];      // sum_{j < n} u_b^(j + 1): the "+ 1" of n tokens
  uint64_t sub_mul[2][32];   // u_b^(16 q)
};

struct HashCarry {
  uint64_t v0, v1, f;
};

struct SegSumOp {
  __device__ HashCarry operator()(const HashCarry& a, const HashCarry& b) const {
    HashCarry r;
    r.f = a.f | b.f;
    r.v0 = b.f ? b.v0 : p61_add(a.v0, b.v0);
    r.v1 = b.f ? b.v1 : p61_add(a.v1, b.v1);
    return r;
  }
};

struct HashArgs {
  const uint32_t* tokens;
  uint64_t n_tok;
  const uint64_t* tok_off;
  const uint64_t* blk_off;
  uint32_t R;
  uint32_t B;
  ulonglong2* keys;
  uint64_t keys_cap;
  const uint64_t* tables;
  const uint32_t* tile_req;
  HashCarry* tile_agg;   // per tile: (request starts inside?, sum of g after the last start)
  uint32_t* tile_lead;   // per tile: blocks before its first request start (keys left normalised)
  DevStatus* st;
  int aligned;
  uint32_t g, tb;       // k_hash_units: units per block, blocks per tile
};

__device__ __forceinline__ uint32_t pad16(uint32_t i) { return i + (i >> 4); }

// 32 x 32 -> 64-bit multiply-add; written in C so the compiler can take the
// constant operand straight from the parameter bank.
__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
  return (uint64_t)a * (uint64_t)b + c;
}

// Sum over the U words wd[M ..] of wd[M + j] u^(j + 1) for both bases, as
// 21-bit limb accumulators.
template <int U, int M, int NW>
__device__ __forceinline__ void unit_sum_3(const uint32_t (&wd)[NW], const HashConsts& c, uint64_t (&acc)[6]) {
  static_assert(M + U <= NW, "unit words out of range");
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t t = wd[j + M];
    acc[0] = mad_wide(t, c.limb[0][0][j], acc[0]);
    acc[1] = mad_wide(t, c.limb[0][1][j], acc[1]);
    acc[2] = mad_wide(t, c.limb[0][2][j], acc[2]);
    acc[3] = mad_wide(t, c.limb[1][0][j], acc[3]);
    acc[4] = mad_wide(t, c.limb[1][1][j], acc[4]);
    acc[5] = mad_wide(t, c.limb[1][2][j], acc[5]);
  }
}

// The same sum with two limbs (31 + 30 bits), exact when every token is
// below 2^27: 16 products of at most 2^58 stay below 2^62.
template <int U, int M, int NW>
__device__ __forceinline__ void unit_sum_2(const uint32_t (&wd)[NW], const HashConsts& c, uint64_t (&acc)[4]) {
  static_assert(M + U <= NW, "unit words out of range");
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t t = wd[j + M];
    acc[0] = mad_wide(t, c.limb2[0][0][j], acc[0]);
    acc[1] = mad_wide(t, c.limb2[0][1][j], acc[1]);
    acc[2] = mad_wide(t, c.limb2[1][0][j], acc[2]);
    acc[3] = mad_wide(t, c.limb2[1][1][j], acc[3]);
  }
}

// Congruent to (a0 + a1 2^31) mod p and below 2^62 + 2^61 + 2^31, for a0 < 2^62
// and a1 < 2^61 (sums of 16 products of a token below 2^27 and a 31- or 30-bit
// limb).
__device__ __forceinline__ uint64_t limbs2_lazy(uint64_t a0, uint64_t a1) {
  return a0 + ((a1 & ((1ULL << 30) - 1)) << 31) + (a1 >> 30);
}

// a b mod p, reduced only below 2^61 + 8, for a < 2^63 + 2^33 and b < p: the
// product is below 2^124 + 2^94, so hi << 3 < 2^63 + 2^33 and the first sum stays
// below 2^64.
__device__ __forceinline__ uint64_t p61_mul_lazy(uint64_t a, uint64_t b) {
  const uint64_t lo = a * b, hi = __umul64hi(a, b);
  const uint64_t r = (lo & kP61) + (lo >> 61) + (hi << 3);
  return (r & kP61) + (r >> 61);
}

// (a0 + a1 2^21 + a2 2^42) mod p for a0, a1, a2 < 2^62 - 2^57 (sums of <= 32 products < 2^53)
__device__ __forceinline__ uint64_t limbs_to_p61(uint64_t a0, uint64_t a1, uint64_t a2) {
  uint64_t x = a0 + ((a1 & ((1ULL << 40) - 1)) << 21) + (a1 >> 40) + ((a2 & ((1ULL << 19) - 1)) << 42) + (a2 >> 19);
  return p61_fold(x);
}

__device__ __forceinline__ uint32_t find_request(const uint64_t* __restrict__ blk_off, uint32_t lo, uint32_t hi,
                                                 uint64_t b) {
  // largest r in [lo, hi] with blk_off[r] <= b (blk_off[lo] <= b holds)
  while (lo < hi) {
    uint32_t mid = (lo + hi + 1) >> 1;
    if (__ldg(&blk_off[mid]) <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Shared second half of the local hash kernels: combine the sub-chunks of each
// block, normalise, segmented sum over the tile, write keys and the tile's
// aggregate.  Every thread of the CTA calls it.
template <int G>
__device__ __forceinline__ void hash_finish(const HashArgs& a, uint32_t tile, uint64_t b0, uint64_t b_end, uint64_t h0,
                                            uint64_t h1, uint32_t k, uint32_t lb, uint32_t s) {
  constexpr uint32_t TB = kHashThreads / G;
  __shared__ uint64_t s_h0[kHashThreads / G], s_h1[kHashThreads / G];
  __shared__ uint32_t s_k[kHashThreads / G];
  __shared__ HashCarry s_w[kHashThreads / 32];
  __shared__ uint32_t s_first_head;
  if (G > 1) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      h0 = p61_add(h0, __shfl_xor_sync(kFull, h0, o));
      h1 = p61_add(h1, __shfl_xor_sync(kFull, h1, o));
    }
  }
  if (G > 1) {  // one value per block: the sub-chunk holding it hands it over
    if (s == 0) {
      s_h0[lb] = h0;
      s_h1[lb] = h1;
      s_k[lb] = k;
    }
    __syncthreads();
  }

  // ---- phase 2: normalise, segmented sum over requests, denormalise
  const uint32_t t = threadIdx.x;
  const bool valid = t < TB && b0 + t < b_end;
  const uint64_t* T = a.tables;
  HashCarry x{0, 0, 0};
  uint32_t kk = 0;
  if (valid) {
    kk = G > 1 ? s_k[t] : k;
    x.v0 = p61_mul(G > 1 ? s_h0[t] : h0, pow_at(T + 0 * 65536, T + 1 * 65536, kk));
    x.v1 = p61_mul(G > 1 ? s_h1[t] : h1, pow_at(T + 2 * 65536, T + 3 * 65536, kk));
    x.f = kk == 0;
  }
  SegSumOp op;
  const uint32_t lane = t & 31, w = t >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    HashCarry y;
    y.v0 = __shfl_up_sync(kFull, x.v0, d);
    y.v1 = __shfl_up_sync(kFull, x.v1, d);
    y.f = __shfl_up_sync(kFull, x.f, d);
    if (lane >= (uint32_t)d) x = op(y, x);
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  if (w == 0) {
    HashCarry z = lane < kHashThreads / 32 ? s_w[lane] : HashCarry{0, 0, 0};
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      HashCarry y;
      y.v0 = __shfl_up_sync(kFull, z.v0, d);
      y.v1 = __shfl_up_sync(kFull, z.v1, d);
      y.f = __shfl_up_sync(kFull, z.f, d);
      if (lane >= (uint32_t)d) z = op(y, z);
    }
    if (lane < kHashThreads / 32) s_w[lane] = z;  // inclusive over warps
  }
  __syncthreads();
  if (w > 0) x = op(s_w[w - 1], x);
  // Blocks at or after the tile's first request start are final here; the
  // leading blocks still lack the carry from earlier tiles (k_hash_chain).
  if (t == 0) s_first_head = TB;
  __syncthreads();
  if (valid && kk == 0) atomicMin(&s_first_head, t);
  __syncthreads();
  if (valid) a.keys[b0 + t] = make_ulonglong2(x.v0, x.v1);
  if (t == 0) {
    a.tile_agg[tile] = s_w[kHashThreads / 32 - 1];
    const uint32_t nb = (uint32_t)(b_end - b0);
    a.tile_lead[tile] = s_first_head < nb ? s_first_head : nb;
  }
}

template <int G, bool FULL>
__global__ void __launch_bounds__(kHashThreads) k_hash_local(HashArgs a, const __grid_constant__ HashConsts c) {
  grid_dep_sync();
  __shared__ uint32_t s_tok[kWinWords];
  __shared__ uint64_t s_bnd[4];
  constexpr uint32_t TB = kHashThreads / G;

  const uint32_t tile = blockIdx.x;
  const uint64_t N = blocks_live(a.st, a.keys_cap);
  const uint64_t b0 = (uint64_t)tile * TB;
  if (b0 >= N) return;
  const uint64_t b_end = b0 + TB < N ? b0 + TB : N;
  const uint32_t B = a.B;

  if (threadIdx.x == 0) {
    const uint64_t ntiles = (N + TB - 1) / TB;
    const uint32_t r0 = a.tile_req[tile];
    const uint32_t rh = tile + 1 < ntiles ? a.tile_req[tile + 1] : a.R - 1;
    s_bnd[0] = r0;
    s_bnd[1] = find_request(a.blk_off, r0, rh, b_end - 1);
  }
  __syncthreads();
  const uint32_t r_first = (uint32_t)s_bnd[0], r_last = (uint32_t)s_bnd[1];
  const uint64_t t_begin = a.tok_off[r_first] + (uint64_t)B * (b0 - a.blk_off[r_first]);
  const uint64_t t_end = a.tok_off[r_last] + (uint64_t)B * (b_end - a.blk_off[r_last]);
  const uint64_t w0 = a.aligned ? (t_begin & ~3ULL) : t_begin;
  uint64_t w_end = t_end < w0 + kWinTokens ? t_end : w0 + kWinTokens;
  if (w_end > a.n_tok) w_end = a.n_tok;
  __syncthreads();

  // ---- stage the token window
  if (a.aligned) {
    const uint32_t nq = (uint32_t)((w_end - w0 + 3) >> 2);
    for (uint32_t i = threadIdx.x; i < nq; i += kHashThreads) {
      const uint64_t x = w0 + 4ULL * i;
      uint4 v;
      if (x + 3 < a.n_tok) {
        v = __ldcs(reinterpret_cast<const uint4*>(a.tokens + x));
      } else {
        v.x = x < a.n_tok ? a.tokens[x] : 0u;
        v.y = x + 1 < a.n_tok ? a.tokens[x + 1] : 0u;
        v.z = x + 2 < a.n_tok ? a.tokens[x + 2] : 0u;
        v.w = 0u;
      }
      const uint32_t o = pad16(4 * i);
      s_tok[o] = v.x;
      s_tok[o + 1] = v.y;
      s_tok[o + 2] = v.z;
      s_tok[o + 3] = v.w;
    }
  } else {
    const uint32_t n = (uint32_t)(w_end - w0);
    for (uint32_t i = threadIdx.x; i < n; i += kHashThreads) s_tok[pad16(i)] = a.tokens[w0 + i];
  }
  __syncthreads();

  // ---- phase 1: 16-token sub-chunks
  const uint32_t lb = threadIdx.x / G, s = threadIdx.x % G;
  const uint64_t b = b0 + lb;
  uint64_t h0 = 0, h1 = 0;
  uint32_t k = 0;
  if (b < b_end) {
    const uint32_t r = find_request(a.blk_off, r_first, r_last, b);
    k = (uint32_t)(b - a.blk_off[r]);
    const uint32_t first = 16 * s;  // block offset of this chunk's token 0
    const uint32_t nval = first < B ? (B - first < 16 ? B - first : 16) : 0u;  // tokens of the block in the chunk
    const uint64_t bstart = a.tok_off[r] + (uint64_t)B * k;
    uint64_t a00 = 0, a01 = 0, a02 = 0, a10 = 0, a11 = 0, a12 = 0;
    const uint64_t x0 = bstart + first;
    const bool in_win = FULL && x0 >= w0 && x0 + 16 <= w_end;
    if (in_win) {
      const uint32_t rel = (uint32_t)(x0 - w0);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const uint64_t t = s_tok[pad16(rel + j)];
        a00 += t * c.limb[0][0][j];
        a01 += t * c.limb[0][1][j];
        a02 += t * c.limb[0][2][j];
        a10 += t * c.limb[1][0][j];
        a11 += t * c.limb[1][1][j];
        a12 += t * c.limb[1][2][j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (FULL || (uint32_t)j < nval) {
          const uint64_t x = x0 + (uint64_t)j;
          uint64_t t;
          if (x >= w0 && x < w_end)
            t = s_tok[pad16((uint32_t)(x - w0))];
          else
            t = x < a.n_tok ? a.tokens[x] : 0u;
          a00 += t * c.limb[0][0][j];
          a01 += t * c.limb[0][1][j];
          a02 += t * c.limb[0][2][j];
          a10 += t * c.limb[1][0][j];
          a11 += t * c.limb[1][1][j];
          a12 += t * c.limb[1][2][j];
        }
      }
    }
    h0 = p61_add(limbs_to_p61(a00, a01, a02), c.csum[0][FULL ? 16 : nval]);
    h1 = p61_add(limbs_to_p61(a10, a11, a12), c.csum[1][FULL ? 16 : nval]);
    if (G > 1 && s > 0) {
      h0 = p61_mul(h0, c.sub_mul[0][s]);
      h1 = p61_mul(h1, c.sub_mul[1][s]);
    }
  }
  hash_finish<G>(a, tile, b0, b_end, h0, h1, k, lb, s);
}

// B = g U with U = 16, 12 or 8 tokens per unit, tokens at any 4-byte
// alignment.  With units numbered through a request (unit e of it covers its
// tokens [U e, U e + U)) the key of a block is the sum over the units up to
// its last one of h_e u^(U e), so units are hashed and summed alike and only
// every g-th sum is written.
//
// One warp per tile of tb blocks (tb g <= 32 PER units, tb a power of two), no
// CTA barrier anywhere:
//   units   32 at a time, one per lane: its 16-byte loads (a unit that does
//           not start on a 16-byte boundary takes its last words from the next
//           lane), the limb products, one multiplication by u^(U e); the
//           result to shared memory
//   sums    PER consecutive units per lane (8, 9 or 11: launch_units): a serial
//           sum that starts anew where a request starts, one segmented scan over
//           the lanes, and the canonical residues back to shared memory
//   store   the block ends, coalesced
// What bounds it: L1's data path (73% busy), the pipe that multiplies (67%),
// issue (58%) and DRAM (75% of a copy's rate) together.  The form before this
// one gave each of 256 threads one block and ran a warp scan, a scan over the warps and
// the exchange of request starts for every block, with four CTA barriers: 562
// instructions a block, of which the products are 64.
// Measured (keys and tokens over the time; the form before in brackets): 735
// us or 5.2 TB/s on 763M tokens of the agentic trace [3.7 TB/s on the whole
// one], 163 us on the chat trace [214], 679 us on 724M tokens in blocks of 64
// that start at an odd word [1,675], 77 us on 55M tokens in blocks of 24 [223].
// It pays for every instruction of a round: 844 us with the limb sums folded
// before the multiplication, bounds tested per lane, lanes past the tile's end
// masked and 64-bit slot and power addresses, 753 without.  18 CTAs an SM are the
// best number: 846 us with 12, 790 with 14, 753 with 16, 962 with 20 (48
// registers) and 1,054 with 21; the sums one word at a time, in half the
// registers, took 743 with 18 and 959 with 20.  Not kept either: 22 warps with
// the tokens staged in shared memory a round ahead (30% longer), the products on
// the tensor cores (exact, as byte products; 36 to 47%: the bookkeeping around
// them is more), a separate path for tiles inside one request with the next
// round's tokens loaded ahead (as long on the agentic trace, a third longer on the
// chat trace, where both paths' code competes for the instruction cache), and the
// sums without the starts' tests where a tile has none (1.4% less there, 1.8% more
// on the chat trace).
constexpr uint32_t kUnitWarps = 2;  // per CTA: small, so that few tiles still spread over the SMs
constexpr uint32_t kUnitThreads = 32 * kUnitWarps;
// PER units per lane in the sums, 32 PER per tile at most.  A slot of padding per
// lane's units where PER is even, so that the lanes' slots lie an odd number apart.
template <int PER>
__host__ __device__ constexpr uint32_t unit_slot(uint32_t v) {
  return PER % 2 ? v : v + v / PER;
}

// x mod p for any 64-bit x.
__device__ __forceinline__ uint64_t p61_canon(uint64_t x) {
  const uint64_t y = (x & kP61) + (x >> 61);  // at most p + 7
  return y >= kP61 ? y - kP61 : y;
}
__device__ __forceinline__ uint64_t p61_part(uint64_t x) { return (x & kP61) + (x >> 61); }

// h of a unit whose first token is word M of wd: below 2^63 + 2^32.
template <int U, int M, bool WIDE, int NW>
__device__ __forceinline__ void unit_hash(const uint32_t (&wd)[NW], const HashConsts& c, uint64_t& h0, uint64_t& h1) {
  if (WIDE) {
    uint64_t acc[6] = {0, 0, 0, 0, 0, 0};
    unit_sum_3<U, M>(wd, c, acc);
    h0 = p61_add(limbs_to_p61(acc[0], acc[1], acc[2]), c.csum[0][U]);
    h1 = p61_add(limbs_to_p61(acc[3], acc[4], acc[5]), c.csum[1][U]);
  } else {
    uint64_t acc[4] = {0, 0, 0, 0};
    unit_sum_2<U, M>(wd, c, acc);
    h0 = limbs2_lazy(acc[0], acc[1]) + c.csum[0][U];
    h1 = limbs2_lazy(acc[2], acc[3]) + c.csum[1][U];
  }
}

__device__ __forceinline__ int64_t shfl_i64(int64_t v, uint32_t src) {
  return (int64_t)__shfl_sync(kFull, (unsigned long long)v, src);
}

// The sums of a tile: slot[v] (units' values below 2^61 + 8) becomes the
// canonical sum of the values since the last request start.  `mine` are the
// starts among this lane's PER units, `opens` the lanes that have one.  (Slots
// past the tile's last unit hold anything: sums only reach later units.)
template <int PER>
__device__ __forceinline__ void unit_sums(ulonglong2* slot, uint32_t lane, uint32_t mine, uint32_t opens) {
  uint64_t p0[PER], p1[PER];
  uint64_t s0 = 0, s1 = 0;
  slot += unit_slot<PER>(PER * lane);
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const ulonglong2 t = slot[j];
    if ((mine >> j) & 1u) s0 = s1 = 0;
    s0 += t.x;
    s1 += t.y;
    p0[j] = s0;  // below 5 2^61 + 64
    p1[j] = s1;
    if (j % 4 == 3 && j + 1 < PER) {
      s0 = p61_part(s0);
      s1 = p61_part(s1);
    }
  }
  s0 = p61_part(s0);
  s1 = p61_part(s1);
  // segmented scan over the lanes; from values below 2^61 + 8 two plain steps
  // stay below 2^63 + 32, so a fold every other step keeps sums below 2^64
  const uint32_t upto = opens & (lanemask_lt() | (1u << lane));
  const uint32_t seg = upto ? 31u - __clz(upto) : 0u;  // the sum reaches back to this lane
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t y0 = __shfl_up_sync(kFull, s0, d), y1 = __shfl_up_sync(kFull, s1, d);
    if (lane >= seg + (uint32_t)d) {
      s0 += y0;
      s1 += y1;
    }
    if (d == 2 || d == 8) {
      s0 = p61_part(s0);
      s1 = p61_part(s1);
    }
  }
  uint64_t c0 = __shfl_up_sync(kFull, s0, 1), c1 = __shfl_up_sync(kFull, s1, 1);
  c0 = lane ? p61_part(c0) : 0;
  c1 = lane ? p61_part(c1) : 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if ((mine >> j) & 1u) c0 = c1 = 0;  // the carry ends at the lane's first start
    slot[j] = make_ulonglong2(p61_canon(p0[j] + c0), p61_canon(p1[j] + c1));
  }
}

// One tile, by one warp.  WIDE = false: two-limb products, exact while every
// token is below 2^27 (any vocabulary in use); a tile that holds a larger one
// writes nothing and is left to hash_units_wide.  WIDE = true: three-limb
// products, exact for every 32-bit token.
template <int U, int PER, bool WIDE>
__device__ __forceinline__ bool hash_units_tile(const HashArgs& a, const HashConsts& c, uint32_t tile, uint64_t N,
                                                ulonglong2* slot, uint32_t* starts) {
  constexpr int NV = U / 4;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t b0 = (uint64_t)tile * a.tb;
  if (b0 >= N) return false;
  const uint32_t nb = N - b0 < a.tb ? (uint32_t)(N - b0) : a.tb, nu = nb * a.g;
  const uint64_t ntiles = (N + a.tb - 1) / a.tb;
  const uint32_t r_first = a.tile_req[tile];
  const uint32_t r_last = tile + 1 < ntiles ? a.tile_req[tile + 1] : a.R - 1;  // the last request meeting the tile
  // the token array from the 16-byte boundary at or below its start
  const uint32_t mis = (uint32_t)(reinterpret_cast<uintptr_t>(a.tokens) >> 2) & 3u;
  const uint32_t* base = a.tokens - mis;
  const uint64_t n_word = a.n_tok + mis;
  // A window of 32 requests from rw, one per lane: unit v of the tile that
  // lies in one of them is unit v + e0 of the request and starts at word
  // x0 + U v.  `past` is the first unit after the window.
  uint32_t rw = r_first, wn = 0;
  int64_t e0 = 0, x0 = 0, past = 0;
  auto window = [&]() {
    wn = r_last - rw + 1 < 32 ? r_last - rw + 1 : 32;
    const uint32_t r = rw + (lane < wn ? lane : wn - 1);
    e0 = ((int64_t)b0 - (int64_t)a.blk_off[r]) * (int64_t)a.g;
    x0 = (int64_t)(a.tok_off[r] + mis) + U * e0;
    past = ((int64_t)a.blk_off[rw + wn] - (int64_t)b0) * (int64_t)a.g;
  };
  window();
  const bool one = r_first == r_last;
  bool big = false;
  ulonglong2* out = slot + unit_slot<PER>(lane);
#pragma unroll 1
  for (uint32_t v0 = 0; v0 < nu; v0 += 32) {
    const uint32_t v = v0 + lane;
    const bool live = v < nu;
    const uint32_t vc = live ? v : nu - 1;  // a lane past the tile does its last unit again, which nobody reads
    int64_t e = e0, x = x0;                 // of this lane's unit
    if (!one) {
      const uint32_t last = nu - v0 < 32 ? nu - 1 : v0 + 31;
      if (past <= (int64_t)last) {  // move the window to the request of this round's first unit
        const uint32_t in = __popc(__ballot_sync(kFull, lane < wn && -e0 <= (int64_t)v0));
        rw = past <= (int64_t)v0 ? find_request(a.blk_off, rw, r_last, b0 + v0 / a.g) : rw + (in ? in - 1 : 0);
        window();
      }
      if (past > (int64_t)last) {
        uint32_t idx = 0;
        for (uint32_t i = 1; i < wn; ++i) {
          const int64_t st = -shfl_i64(e0, i);
          if (st > (int64_t)last) break;
          if (st <= (int64_t)vc) idx = i;
        }
        e = shfl_i64(e0, idx);
        x = shfl_i64(x0, idx);
      } else {  // more requests than the window holds (many without blocks)
        const uint32_t r = find_request(a.blk_off, rw, r_last, b0 + vc / a.g);
        e = ((int64_t)b0 - (int64_t)a.blk_off[r]) * (int64_t)a.g;
        x = (int64_t)(a.tok_off[r] + mis) + U * e;
      }
    }
    e += vc;
    x += (int64_t)U * vc;
    const uint32_t st = __ballot_sync(kFull, live && e == 0);  // units that open a request
    if (lane == 0) starts[v0 >> 5] = st;
    // its words: NV aligned vectors, and for a unit that starts m words into
    // the first the next vector's m words, which the next lane holds if its
    // unit follows on
    const uint32_t m = (uint32_t)x & 3u;
    const uint64_t x4 = (uint64_t)x & ~3ULL;
    const bool follows = lane < 31 && v + 1 < nu && !((st >> (lane + 1)) & 1u);  // the next lane has the next vector
    // A request with blocks ends at or before the array's end, and so do the
    // unit's NV vectors; the first may begin before the array if that does not
    // begin on a boundary itself.
    bool inside = true;
    if (mis) inside = __all_sync(kFull, x4 != 0);
    uint32_t wd[U + 4];
    uint4 nx = make_uint4(0, 0, 0, 0);
    if (inside) {
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        const uint4 t = __ldcs(reinterpret_cast<const uint4*>(base + x4) + q);
        wd[4 * q] = t.x;
        wd[4 * q + 1] = t.y;
        wd[4 * q + 2] = t.z;
        wd[4 * q + 3] = t.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < U; ++q) wd[q] = x4 + q >= mis ? base[x4 + q] : 0u;
    }
    if (m != 0 && !follows) {
      const uint64_t y = x4 + U;
      if (y + 4 <= n_word) {
        nx = __ldcs(reinterpret_cast<const uint4*>(base + y));
      } else {
        nx.x = y < n_word ? base[y] : 0u;
        nx.y = y + 1 < n_word ? base[y + 1] : 0u;
        nx.z = y + 2 < n_word ? base[y + 2] : 0u;
      }
    }
    // the powers go out with the tokens
    const uint64_t* T = a.tables;
    const uint32_t e_lo = (uint32_t)e & 0xFFFFu, e_hi = (uint32_t)e >> 16;  // e < 2^32 (unit_tokens)
    uint64_t w0 = __ldg(&T[e_lo]), w1 = __ldg(&T[2 * 65536 + e_lo]);
    if (e_hi) {
      w0 = p61_mul(w0, __ldg(&T[65536 + e_hi]));
      w1 = p61_mul(w1, __ldg(&T[3 * 65536 + e_hi]));
    }
    if (__any_sync(kFull, m != 0)) {
      const uint32_t n0 = __shfl_down_sync(kFull, wd[0], 1), n1 = __shfl_down_sync(kFull, wd[1], 1),
                     n2 = __shfl_down_sync(kFull, wd[2], 1);
      if (follows) nx = make_uint4(n0, n1, n2, 0u);
    }
    wd[U] = nx.x;
    wd[U + 1] = nx.y;
    wd[U + 2] = nx.z;
    wd[U + 3] = 0;
    if (!WIDE) {  // words around the unit only widen the test
      uint32_t any = 0;
#pragma unroll
      for (int q = 0; q < U + 3; ++q) any |= wd[q];
      big |= (any >> 27) != 0;
    }
    uint64_t h0, h1;
    switch (m) {
      case 0: unit_hash<U, 0, WIDE>(wd, c, h0, h1); break;
      case 1: unit_hash<U, 1, WIDE>(wd, c, h0, h1); break;
      case 2: unit_hash<U, 2, WIDE>(wd, c, h0, h1); break;
      default: unit_hash<U, 3, WIDE>(wd, c, h0, h1); break;
    }
    *out = make_ulonglong2(p61_mul_lazy(h0, w0), p61_mul_lazy(h1, w1));
    static_assert(PER % 2 || 32 % PER == 0, "32 units further, the padding has grown by whole lanes");
    out += PER % 2 ? 32 : 32 + 32 / PER;  // unit_slot(v + 32)
  }
  if (!WIDE && __any_sync(kFull, big)) return true;
  __syncwarp();
  // ---- sums: this lane's units PER lane .. PER lane + PER - 1 (values below 2^61 + 8)
  const uint32_t rounds = (nu + 31) / 32;
  const uint32_t at = PER * lane, sw = at >> 5;  // the lane's starts begin at bit `at`
  uint32_t mine = sw < rounds ? starts[sw] >> (at & 31) : 0u;
  if (32 % PER != 0 && (at & 31) + PER > 32 && sw + 1 < rounds) mine |= starts[sw + 1] << (32 - (at & 31));
  mine &= (1u << PER) - 1u;
  const uint32_t opens = __ballot_sync(kFull, mine != 0);
  unit_sums<PER>(slot, lane, mine, opens);
  __syncwarp();
  for (uint32_t i = lane; i < nb; i += 32) a.keys[b0 + i] = slot[unit_slot<PER>((i + 1) * a.g - 1)];
  // the tile's aggregate for the carry: its last unit's sum since its request's
  // start, and whether a request starts in the tile; and the blocks before the
  // tile's first request start
  if (lane == 0) {
    const ulonglong2 t = slot[unit_slot<PER>(nu - 1)];
    uint32_t lead = nb;
    for (int q = (int)rounds - 1; q >= 0; --q)
      if (starts[q]) lead = (32 * q + __ffs(starts[q]) - 1) / a.g;
    a.tile_agg[tile] = HashCarry{t.x, t.y, opens != 0};
    a.tile_lead[tile] = lead;
  }
  return false;
}

// Kept out of line, so that the three-limb code is not part of every tile's
// path (nor its registers of it).
template <int U, int PER>
__device__ __noinline__ void hash_units_wide(const HashArgs& a, const HashConsts& c, uint32_t tile, uint64_t N,
                                             ulonglong2* slot, uint32_t* starts) {
  hash_units_tile<U, PER, true>(a, c, tile, N, slot, starts);
}

template <int U, int PER>
__global__ void __launch_bounds__(kUnitThreads, PER == 11 ? 16 : 18) k_hash_units(const __grid_constant__ HashArgs a,
                                                                 const __grid_constant__ HashConsts c) {
  grid_dep_sync();
  __shared__ ulonglong2 s_slot[kUnitWarps][unit_slot<PER>(32 * PER - 1) + 1];
  __shared__ uint32_t s_starts[kUnitWarps][PER];
  const uint32_t w = threadIdx.x >> 5, tile = blockIdx.x * kUnitWarps + w;
  const uint64_t N = blocks_live(a.st, a.keys_cap);
  if (hash_units_tile<U, PER, false>(a, c, tile, N, s_slot[w], s_starts[w])) {
    __syncwarp();
    hash_units_wide<U, PER>(a, c, tile, N, s_slot[w], s_starts[w]);
  }
}

// The segmented sum of the aggregates of the tiles before t0, back to (and
// including) the nearest one where a request starts, by one warp, 32 tiles a
// round.  All aggregates exist before the kernel starts, so nothing waits.
__device__ __forceinline__ HashCarry carry_into(const HashCarry* __restrict__ tile_agg, uint32_t t0, uint32_t lane) {
  HashCarry c{0, 0, 0};
  for (int64_t base = (int64_t)t0 - 1; base >= 0; base -= 32) {
    const int64_t idx = base - (int64_t)lane;
    HashCarry g{0, 0, 0};
    if (idx >= 0) g = tile_agg[idx];
    const uint32_t heads = __ballot_sync(kFull, idx >= 0 && g.f);
    const uint32_t first = heads ? (uint32_t)(__ffs(heads) - 1) : 31u;
    uint64_t v0 = lane <= first ? g.v0 : 0, v1 = lane <= first ? g.v1 : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v0 = p61_add(v0, __shfl_xor_sync(kFull, v0, o));
      v1 = p61_add(v1, __shfl_xor_sync(kFull, v1, o));
    }
    c.v0 = p61_add(c.v0, v0);
    c.v1 = p61_add(c.v1, v1);
    if (heads) break;
  }
  return c;
}
// The carry of every tile of a warp's PER (lane q: tile t0 + q) from the one into
// the first: a segmented scan of their aggregates over the lanes.
template <int PER>
__device__ __forceinline__ HashCarry lane_carries(const HashCarry* __restrict__ tile_agg, uint32_t t0, uint64_t live,
                                                  const HashCarry& cin, uint32_t lane) {
  const SegSumOp op;
  const uint32_t t = t0 + lane;
  HashCarry g{0, 0, 0};
  if (lane < PER && t < live) g = tile_agg[t];
#pragma unroll
  for (int o = 1; o < PER; o <<= 1) {  // inclusive segmented sums over lanes 0 .. PER - 1
    HashCarry y;
    y.v0 = __shfl_up_sync(kFull, g.v0, o);
    y.v1 = __shfl_up_sync(kFull, g.v1, o);
    y.f = __shfl_up_sync(kFull, g.f, o);
    if (lane >= (uint32_t)o) g = op(y, g);
  }
  HashCarry before;  // this warp's tiles before tile t
  before.v0 = __shfl_up_sync(kFull, g.v0, 1);
  before.v1 = __shfl_up_sync(kFull, g.v1, 1);
  before.f = __shfl_up_sync(kFull, g.f, 1);
  if (lane == 0) before = HashCarry{0, 0, 0};
  return op(cin, before);
}

// The carry of every tile (carry_into) added to its leading blocks, the tail of a
// request that started earlier.  A warp takes PER consecutive tiles, 256 blocks or
// fewer: PER = 8 where a tile holds at most 32.  (With a warp per tile 1.5M blocks
// of 272 tokens, eight to a tile, took 56 us, so, sixteen to a tile, 14.)
constexpr int kChainWarps = 8;
template <int PER>
__global__ void __launch_bounds__(kChainWarps * 32) k_hash_chain(ulonglong2* __restrict__ keys,
                                                                 const HashCarry* __restrict__ tile_agg,
                                                                 const uint32_t* __restrict__ tile_lead, uint32_t TB,
                                                                 const DevStatus* st, uint64_t keys_cap) {
  grid_dep_sync();
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t t0 = (blockIdx.x * kChainWarps + (threadIdx.x >> 5)) * PER;
  const uint64_t N = blocks_live(st, keys_cap);
  const uint64_t b0 = (uint64_t)t0 * TB, live = (N + TB - 1) / TB;
  if (t0 >= live) return;
  const uint32_t t = t0 + lane;
  const uint32_t lead = lane < PER && t > 0 && t < live ? tile_lead[t] : 0u;
  if (!__any_sync(kFull, lead != 0)) return;
  HashCarry c{0, 0, 0};
  if (__shfl_sync(kFull, lead, 0)) c = carry_into(tile_agg, t0, lane);
  if (PER == 1) {
    const uint32_t n = __shfl_sync(kFull, lead, 0);
    for (uint32_t i = lane; i < n; i += 32) {
      if (!in_bounds(st, b0 + i, keys_cap)) return;
      const ulonglong2 k = keys[b0 + i];
      keys[b0 + i] = make_ulonglong2(p61_add(k.x, c.v0), p61_add(k.y, c.v1));
    }
    return;
  }
  c = lane_carries<PER>(tile_agg, t0, live, c, lane);
  const uint32_t shift = 31 - __clz(TB);
  for (uint32_t j = lane; j < PER * TB; j += 32) {  // whole warps: TB is 4 or more
    const uint32_t q = j >> shift;
    const uint32_t n = __shfl_sync(kFull, lead, q);
    const uint64_t c0 = __shfl_sync(kFull, c.v0, q), c1 = __shfl_sync(kFull, c.v1, q);
    if ((j & (TB - 1)) < n && in_bounds(st, b0 + j, keys_cap)) {
      const ulonglong2 k = keys[b0 + j];
      keys[b0 + j] = make_ulonglong2(p61_add(k.x, c0), p61_add(k.y, c1));
    }
  }
}

// The same carries as k_hash_chain, left for the keys' reader instead of
// added to the keys (a pipeline that does not return the keys saves the
// pass over them): carry[t] and lead[t] per tile, 0 where no key needs one.
// A warp takes kCarryPer consecutive tiles: the carry into the first from a
// look-back over the aggregates before it (all written, so nothing waits),
// then a segmented scan of its own tiles' aggregates across kCarryPer lanes.
constexpr int kCarryPer = 8;
__global__ void __launch_bounds__(kChainWarps * 32) k_hash_carry(const HashCarry* __restrict__ tile_agg,
                                                                 const uint32_t* __restrict__ tile_lead, uint32_t TB,
                                                                 const DevStatus* st, uint64_t keys_cap,
                                                                 uint32_t ntiles, ulonglong2* __restrict__ carry,
                                                                 uint32_t* __restrict__ lead_out) {
  grid_dep_sync();
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t t0 = (blockIdx.x * kChainWarps + (threadIdx.x >> 5)) * kCarryPer;
  if (t0 >= ntiles) return;
  const uint64_t N = blocks_live(st, keys_cap);
  const uint64_t live = (N + TB - 1) / TB;  // tiles that hold blocks
  HashCarry c{0, 0, 0};
  if (t0 < live) c = carry_into(tile_agg, t0, lane);
  c = lane_carries<kCarryPer>(tile_agg, t0, live, c, lane);
  const uint32_t t = t0 + lane;
  if (lane < kCarryPer && t < ntiles) {
    const uint64_t b0 = (uint64_t)t * TB;
    const uint32_t lead = (b0 >= N || t == 0) ? 0u : tile_lead[t];
    carry[t] = lead ? make_ulonglong2(c.v0, c.v1) : make_ulonglong2(0, 0);
    lead_out[t] = lead;
  }
}

// Units per lane: 8, but 9 or 11 where a power of two of blocks is more than 256
// units and up to 288 or 352 (half of them would fill 256 badly: a tile's sums and
// its last, partial round cost as much for few units).  400M tokens: B = 144 456
// us in tiles of 144 units, 380 in 288; B = 272 479 and 397; B = 80 422 in 160 and
// 393 in 320; B = 336 446 in 168 and 397 in 336.  11 per lane take 16 CTAs per SM
// (with 18, whose registers spill, B = 336 took 418); 9 take 18 (B = 272: 402 with
// 16).
constexpr uint32_t kUnitPer = 8, kUnitPerMost = 11;

template <int U>
void launch_units(uint32_t tiles, cudaStream_t s, const HashArgs& a, const HashConsts& c) {
  const uint32_t grid = ceil_div_u32(tiles, kUnitWarps), units = a.tb * a.g;
  if (units <= 32 * kUnitPer)
    PTC_KERNEL("k_hash_units", s, (k_hash_units<U, kUnitPer>), grid, kUnitThreads, 0, a, c);
  else if (units <= 32 * 9)
    PTC_KERNEL("k_hash_units", s, (k_hash_units<U, 9>), grid, kUnitThreads, 0, a, c);
  else
    PTC_KERNEL("k_hash_units", s, (k_hash_units<U, kUnitPerMost>), grid, kUnitThreads, 0, a, c);
}

template <int G>
void launch_hash(uint32_t grid, cudaStream_t s, const HashArgs& a, const HashConsts& c, bool full) {
  if (full)
    PTC_KERNEL("k_hash_local", s, (k_hash_local<G, true>), grid, kHashThreads, 0, a, c);
  else
    PTC_KERNEL("k_hash_local", s, (k_hash_local<G, false>), grid, kHashThreads, 0, a, c);
}

// Tokens per unit of k_hash_units, or 0 for a trace that k_hash_local takes.
// Units are whole vectors of four tokens, so that the units of a request share
// their alignment; the larger the unit, the fewer multiplications and sums per
// token.  A unit's place in its request is a 32-bit exponent: where a request
// could hold 2^32 units (34 billion tokens or more), blocks are counted instead,
// of which no trace has that many.
uint32_t unit_tokens(uint32_t B, uint64_t n_tok) {
  const uint32_t U = B % 16 == 0 ? 16 : B % 12 == 0 ? 12 : B % 8 == 0 ? 8 : 0;
  return U && n_tok / U < 1ULL << 32 ? U : 0;
}

uint32_t chunks_per_block(uint32_t B) {  // G: power of two >= ceil(B / 16)
  uint32_t need = (B + 15) / 16, g = 1;
  while (g < need) g <<= 1;
  return g;
}

// Blocks per hash tile for n_tok tokens, a power of two: 256 or fewer that make up
// to 352 units (launch_units) for k_hash_units, one CTA's kHashThreads / G for
// k_hash_local.  With few blocks a tile of units is cut down to 64 while there are
// fewer tiles than kUnitFewTiles, 16 warps on each of the GPU's 152 SMs (36 fit):
// a warp takes its rounds of 32 units one after another, and a window of 127K
// blocks took 20 us in tiles of 256, 13 in tiles of 64.  (A constant, as the size
// of the workspace follows from it, which callers may ask for without a GPU.)
constexpr uint32_t kUnitFewTiles = 16 * 152;
uint32_t tile_blocks(uint32_t B, uint64_t n_tok) {
  // a block is at most 512 / 8 units, or 32 chunks
  static_assert(PTC_MAX_BLOCK_SIZE / 8 * kCarryTileMin <= 32 * kUnitPer && 32 * kCarryTileMin <= kHashThreads,
                "tiles without the cut below hold kCarryTileMin blocks or more");
  const uint32_t U = unit_tokens(B, n_tok);
  const uint64_t nb = n_tok / B;
  if (!U) return kHashThreads / chunks_per_block(B);
  const uint32_t g = B / U;
  uint32_t tb = 32 * kUnitPer;
  while (tb * g > 32 * kUnitPerMost) tb >>= 1;
  while (tb > 1 && tb * g > 64 && nb / tb < kUnitFewTiles) tb >>= 1;
  return tb;
}

struct HashLayout {
  DevStatus* st;
  uint64_t* lb_off;
  HashCarry* tile_agg;
  uint32_t* tile_lead;
  uint64_t* tables;
  uint32_t* tile_req;
  uint64_t hash_tiles;
  size_t zero_bytes;
  size_t total;
};

HashLayout hash_layout(void* ws, uint32_t n_req, uint64_t n_tok, uint32_t B, uint64_t keys_cap) {
  HashLayout L;
  Carver cv(ws);
  const uint32_t off_tiles = ceil_div_u32(n_req, kOffTile) + 1;
  const uint64_t nb = n_tok / B < keys_cap ? n_tok / B : keys_cap;
  const uint32_t tb = tile_blocks(B, n_tok);
  const uint32_t hash_tiles = ceil_div_u32(nb, tb) + 1;
  L.st = cv.take<DevStatus>(1);
  L.lb_off = cv.take<uint64_t>(off_tiles);
  L.zero_bytes = cv.off;
  L.tile_agg = cv.take<HashCarry>(hash_tiles);
  L.tile_lead = cv.take<uint32_t>(hash_tiles);
  L.tables = cv.take<uint64_t>(4 * 65536);
  L.tile_req = cv.take<uint32_t>(hash_tiles + 1);
  L.hash_tiles = hash_tiles;
  L.total = cv.bytes();
  return L;
}

}  // namespace
}  // namespace ptc

using namespace ptc;

size_t ptc::hash_lb_words(uint32_t n_req) { return ceil_div_u32(n_req, kOffTile) + 1; }

uint64_t ptc::hash_carry_tiles(uint64_t n_tok, uint32_t block_size) {
  if (block_size == 0) block_size = 1;
  return ceil_div_u32(n_tok / block_size, tile_blocks(block_size, n_tok)) + 1;
}

extern "C" size_t ptc_hash_blocks_workspace_bytes(uint32_t n_req, uint64_t n_tok, uint32_t block_size) {
  if (block_size == 0) block_size = 1;
  return hash_layout(nullptr, n_req, n_tok, block_size, ~0ULL).total;
}

ptc_status ptc::hash_impl(const uint32_t* tokens, uint64_t n_tok, const uint64_t* req_tok_off,
                         const int64_t* req_ts_us, uint32_t n_req, uint32_t block_size, uint64_t seed,
                         ptc_u128* keys_out, uint64_t keys_cap, uint64_t* req_blk_off_out,
                         uint64_t* n_access_host_out, void* ws, size_t ws_bytes, cudaStream_t s, DevStatus* lent,
                         uint64_t* lent_lb, KeyCarry* carry, const uint32_t* ses, uint32_t n_session) {
  if (block_size < 1 || block_size > PTC_MAX_BLOCK_SIZE) return PTC_ERR_INVALID_ARG;
  if (req_tok_off == nullptr || req_blk_off_out == nullptr || n_access_host_out == nullptr)
    return PTC_ERR_INVALID_ARG;
  if (n_tok > 0 && tokens == nullptr) return PTC_ERR_INVALID_ARG;
  if (keys_cap > 0 && keys_out == nullptr) return PTC_ERR_INVALID_ARG;
  const HashLayout need = hash_layout(nullptr, n_req, n_tok, block_size, ~0ULL);
  if (!ws_ok(ws, ws_bytes, need.total)) return PTC_ERR_WORKSPACE;
  HashLayout L = hash_layout(ws, n_req, n_tok, block_size, ~0ULL);
  *n_access_host_out = 0;
  if (lent) {
    L.st = lent;
    L.lb_off = lent_lb;
  } else if (begin_call(ws, L.zero_bytes, s) != PTC_OK) {
    return PTC_ERR_CUDA;
  }
  const uint32_t wait_test = test_wait_polls();
  if (wait_test && fill_async(&L.st->wait_test, wait_test, sizeof(uint32_t), s) != PTC_OK) return PTC_ERR_CUDA;
  const uint32_t tb = tile_blocks(block_size, n_tok), U = unit_tokens(block_size, n_tok);
  if (carry) carry->tile_blocks = tb;  // the keys' reader looks carries up whether there are keys or not
  if (n_req == 0) {
    if (fill_async(req_blk_off_out, 0u, sizeof(uint64_t), s) != PTC_OK) return PTC_ERR_CUDA;
    if (lent) return cudaGetLastError() == cudaSuccess ? PTC_OK : PTC_ERR_CUDA;
    DevStatus h;
    return end_call(L.st, s, &h);
  }
  const uint32_t G = chunks_per_block(block_size);
  const bool aligned = (((uintptr_t)tokens) & 15) == 0;
  // seeded bases and their derived constants
  PowArgs pw;
  HashConsts hc;
  for (int b = 0; b < 2; ++b) {
    const uint64_t u = 2 + splitmix64_at(seed, (uint64_t)b) % (kP61 - 3);
    const uint64_t uU = p61_pow(u, U ? U : block_size);
    pw.base[b * 2 + 0] = uU;
    pw.base[b * 2 + 1] = p61_pow(uU, 65536);
    uint64_t sum = 0, v = 1;
    hc.csum[b][0] = 0;
    for (int j = 0; j < 16; ++j) {
      v = p61_mul(v, u);
      hc.limb[b][0][j] = (uint32_t)(v & 0x1FFFFF);
      hc.limb[b][1][j] = (uint32_t)((v >> 21) & 0x1FFFFF);
      hc.limb[b][2][j] = (uint32_t)(v >> 42);
      hc.limb2[b][0][j] = (uint32_t)(v & 0x7FFFFFFF);
      hc.limb2[b][1][j] = (uint32_t)(v >> 31);
      sum = p61_add(sum, v);
      hc.csum[b][j + 1] = sum;
    }
    hc.sub_mul[b][0] = 1;
    for (int q = 1; q < 32; ++q) hc.sub_mul[b][q] = p61_mul(hc.sub_mul[b][q - 1], v);  // v = u^16
  }
  const uint64_t reach = n_tok / (U ? U : block_size);  // units of the longest request there can be
  pw.tables = L.tables;
  pw.n_lo = (uint32_t)(reach < 65535 ? reach + 1 : 65536);
  pw.n_hi = (uint32_t)((reach >> 16) < 65535 ? (reach >> 16) + 1 : 65536);
  pw.off_tiles = ceil_div_u32(n_req, kOffTile);
  PTC_KERNEL("k_block_offsets", s, k_block_offsets, pw.off_tiles + ceil_div_u32(pow_chunks(pw), kOffThreads),
             kOffThreads, 0, req_tok_off, req_ts_us, n_req, n_tok, block_size, tb, req_blk_off_out, L.tile_req,
             L.hash_tiles, L.lb_off, L.st, ses, n_session, pw);

  HashArgs a;
  a.tokens = tokens;
  a.n_tok = n_tok;
  a.tok_off = req_tok_off;
  a.blk_off = req_blk_off_out;
  a.R = n_req;
  a.B = block_size;
  a.keys = reinterpret_cast<ulonglong2*>(keys_out);
  a.keys_cap = keys_cap;
  a.tables = L.tables;
  a.tile_req = L.tile_req;
  a.tile_agg = L.tile_agg;
  a.tile_lead = L.tile_lead;
  a.st = L.st;
  a.aligned = aligned;
  a.g = U ? block_size / U : 1;
  a.tb = tb;
  const bool full = block_size == 16 * G;
  const uint64_t nb = n_tok / block_size < keys_cap ? n_tok / block_size : keys_cap;
  const uint32_t grid = ceil_div_u32(nb, tb);
  if (grid > 0) {
    if (U == 16)
      launch_units<16>(grid, s, a, hc);
    else if (U == 12)
      launch_units<12>(grid, s, a, hc);
    else if (U == 8)
      launch_units<8>(grid, s, a, hc);
    else switch (G) {
      case 1: launch_hash<1>(grid, s, a, hc, full); break;
      case 2: launch_hash<2>(grid, s, a, hc, full); break;
      case 4: launch_hash<4>(grid, s, a, hc, full); break;
      case 8: launch_hash<8>(grid, s, a, hc, full); break;
      case 16: launch_hash<16>(grid, s, a, hc, full); break;
      default: launch_hash<32>(grid, s, a, hc, full); break;
    }
    if (carry) {
      PTC_KERNEL("k_hash_carry", s, k_hash_carry, ceil_div_u32(grid, kChainWarps * kCarryPer), kChainWarps * 32, 0, L.tile_agg,
                 L.tile_lead, tb, L.st, keys_cap, grid, carry->carry, carry->lead);
    } else {
      if (tb <= 32 && tb >= kCarryTileMin)
        PTC_KERNEL("k_hash_chain", s, k_hash_chain<8>, ceil_div_u32(grid, kChainWarps * 8), kChainWarps * 32, 0, a.keys,
                   L.tile_agg, L.tile_lead, tb, L.st, keys_cap);
      else
        PTC_KERNEL("k_hash_chain", s, k_hash_chain<1>, ceil_div_u32(grid, kChainWarps), kChainWarps * 32, 0, a.keys,
                   L.tile_agg, L.tile_lead, tb, L.st, keys_cap);
    }
  }
  if (lent) return cudaGetLastError() == cudaSuccess ? PTC_OK : PTC_ERR_CUDA;
  DevStatus h;
  ptc_status rc = end_call(L.st, s, &h);
  *n_access_host_out = h.value[0];
  if (rc != PTC_OK) return rc;
  if (h.value[0] > keys_cap) return PTC_ERR_INVALID_ARG;
  return PTC_OK;
}

extern "C" ptc_status ptc_hash_blocks(const uint32_t* tokens, uint64_t n_tok, const uint64_t* req_tok_off,
                                      const int64_t* req_ts_us, uint32_t n_req, uint32_t block_size, uint64_t seed,
                                      ptc_u128* keys_out, uint64_t keys_cap, uint64_t* req_blk_off_out,
                                      uint64_t* n_access_host_out, void* ws, size_t ws_bytes, void* stream) {
  return ptc::hash_impl(tokens, n_tok, req_tok_off, req_ts_us, n_req, block_size, seed, keys_out, keys_cap,
                        req_blk_off_out, n_access_host_out, ws, ws_bytes, (cudaStream_t)stream, nullptr, nullptr);
}
