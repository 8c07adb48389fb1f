// Tile kernel of the attribution and feature passes (sm_103a).
//
// Work decomposition.  Batch b starts at merge position kTW * b + off[b];
// k_tile_bounds cuts the positions every D and tile t owns the batches whose
// start falls in window t (whole batches, nothing shared with neighbours).
// Warps take tiles round-robin and work alone: no block-wide barrier is taken
// while tiles are processed, so one warp's memory latency is hidden by the
// other warps' arithmetic.  A warp takes its tile in three steps:
//   1. lane j sums requests 8j .. 8j+7 of each 256, a warp scan turns the sums
//      into prefixes (exact integers) in shared memory;
//   2. one lane per batch takes its batch's sums as a difference of two
//      prefixes, then the segment, the per-request constant and T; non-empty
//      batches leave a record and a head bit at their first request;
//   3. one lane per four consecutive requests finds their record from the head
//      bits, attributes them and adds them to the tenants; what is off the
//      common path is listed and worked off 32 at a time.
// So a request costs about the same instructions whatever the batch sizes, and
// no lane idles on a batch's remainder.  The requests are read twice, the
// second time from L1 or L2.  A batch that reaches past a tile's requests is
// walked on its own afterwards: one of more requests than a tile holds comes
// from a queue that k_tile_bounds has filled, so that such batches spread over
// the chip wherever they start (walk_queue); a smaller one by its warp at once,
// or, above kTAlone requests, by the CTA that met it, once its tiles are done (1e6
// Pareto batches: 85 us, 119 if their warps walk them; 1e7: 538 and 600).  All
// sums are exact integers, so results do not depend on the schedule.
//
// What bounds it: instruction issue and the integer pipe (about 148 warp
// instructions per 32 requests), not HBM.  The shape follows from that: 20 warps
// per SM with 96 registers each spill little (24 warps of 80 took 9 % longer,
// 32 of 64 a third), and the largest tile whose shared memory (182 KB) leaves the
// L1 60 KB (tiles of 1,376 positions leave it 28 KB and took 15 % longer, tiles
// of 768 8 %, from their fixed cost).  The loop of step 3 is kept free of calls
// and small enough for the instruction cache (unrolled twice it took a third
// longer).
// Against a kernel that walked one batch per warp (one call, GB300): 1.36e8
// requests in batches of 16 to 256, fp64 shares, 256 tenants, 1,134 us before
// and 840 now; 3.25e7 in batches of 1 to 64, 16 tenants, 583 and 290; 6.5e5, 113
// and 20; 2.6e7 in Pareto batches, 65,536 tenants, 817 and 541; fp32, 4.1e7 in
// batches of 16 to 256, 322 and 224; 5e7 in batches of 4,096, 531 and 407.
#pragma once

#include "lv_step.cuh"
#include "lv_tenant.cuh"

namespace lv {

constexpr int kTThreads = 640;             // threads of a CTA, one CTA per SM (one tenant table)
constexpr int kTWarps = kTThreads / 32;
constexpr int kTW = 8;                     // merge positions a batch takes besides its requests
constexpr int kTDMin = 128;
constexpr int64_t kTAlone = 512;           // requests a warp walks alone where nothing is queued
constexpr int kTBigs = 64;                 // larger batches a CTA keeps for later
constexpr int64_t kQWarp = 4096;           // requests of a queued batch that a warp walks, at most
constexpr int64_t kQTeam = 24576;          // that a team walks
constexpr int kTTeam = 128, kTTeams = kTThreads / kTTeam;
static_assert(3 * kTTeams <= kTBigs, "a turn of the queue fits the list's memory");
constexpr int kTabN = 4096;                // batch sizes of the K table
constexpr uint32_t kTSmall = 1u << 23;     // p and c of a tile on the common path are below this

// A tile's size.  The passes that write only batch features keep no records, so
// their tiles can be twice as large and leave the L1 more.  2.57e8 requests take
// 508 us (6.1 TB/s), 14 us less than with the other passes' shape; tiles of
// 3,256 positions 1 us less still, of 4,064 36 more, 24 warps 22 more, 16 warps 26.
template <int MODE>
struct Geo {
  static constexpr bool kAttr = (MODE & M_ATTR) != 0;
  static constexpr int kD = kAttr ? 1248 : 2496;           // merge positions, at most
  static constexpr int kCap = kAttr ? 1536 : 2560;         // requests, at most
  static constexpr int kNb = kD / kTW;                     // batches, at most
  static constexpr int kRec = kAttr ? kD / (kTW + 1) + 5 : 1;  // non-empty ones, and room to read past the last
  static constexpr int kBlocks = kCap / 256 + 1;           // blocks of 256 requests, one more for a bound at the end
  static constexpr int kWords = kAttr ? kCap / 32 + 1 : 1;
  static_assert(kCap % 256 == 0 && kD + 3 < kCap, "only a tile's last batch can reach past its requests");
  static_assert(!kAttr || kCap <= kTabN, "a tile's batches are in the K table");
};

// A batch's record: its share constant K + A1 + A3 (three words) and the
// biased exponent of word 1's unit << 20; A2 (two words), n << 4 | fast << 3 |
// slow << 2 | segment, and the fourth word of the constant (used off the fast
// path).  fp32 variant: K, a1, a2, a3 as floats in k.
struct TileRec {
  uint4 k, a;
};

// One warp's tile.  pre: per 8 requests {S1, S2, S3 + prefills << 55} of the
// requests before them in their 256; tot: each 256's totals.
template <int MODE>
struct WarpTile {
  using G = Geo<MODE>;
  union {
    alignas(16) uint4 pre[G::kBlocks * 32];
    uint16_t list[G::kCap];  // step 3: requests off the common path
  };
  alignas(16) uint4 tot[G::kBlocks];
  alignas(16) TileRec rec[G::kRec];
  uint32_t bits[G::kWords];  // head bits: a batch starts at this request
  uint16_t rank[G::kWords];  // heads before word w
  uint32_t n_list;         // entries of list
};

template <int MODE>
struct TSmem {
  WarpTile<MODE> tile[kTWarps];
  alignas(16) SegS seg[4];
  alignas(16) SegFix fx[4];
  float cf[4][5];                     // coefficients as float (fp32 variant)
  alignas(16) Sums red[kTWarps];
  alignas(16) int64_t big[kTBigs];    // batches left for the whole CTA
  int n_big;
  unsigned queued[kQClasses];         // batches in the queue
};

// ---------------------------------------------------------------- bounds

// x / D for 0 <= x < 2^44 and 2 <= D < 2^12, with magic = floor((2^64 - 1) / D) + 1.
__device__ __forceinline__ int64_t div_magic(int64_t x, uint64_t magic) {
  return (int64_t)__umul64hi((uint64_t)x, magic);
}

// Lists the warp's batches b0 + k for which bit k of `mask` is set.
template <class V>
__device__ __forceinline__ void queue_add(const TileQueue &q, int cls, uint32_t mask, int64_t b0, int lane) {
  const int own = __popc(mask);
  int end = own;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(kFull, end, d);
    if (lane >= d) end += o;
  }
  const int total = __shfl_sync(kFull, end, 31);
  if (total == 0) return;
  unsigned base = 0;
  if (lane == 0) base = atomicAdd(q.ctr + kQListed + cls, (unsigned)total);
  int64_t i = q.at[cls] + __shfl_sync(kFull, base, 0) + end - own;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if ((mask >> k) & 1u) {
      if (i < q.at[cls + 1]) static_cast<V *>(q.list)[i] = (V)(b0 + k);  // always, for valid offsets
      ++i;
    }
}

// part[t] = the first batch whose start position kTW * b + off[b] is at least
// t * D, for t in [0, n_tiles); part[n_tiles] = n_batch.  Batch b writes the t
// in (f(b-1) / D, f(b) / D], so every entry is written once.  Checks the
// offsets, and queues the batches of more than `most` requests, which no tile
// holds.  HBM-bound: 8 B per batch; four batches per thread from two 16-byte
// loads, and the divisions are multiplications (1e7 batches take 30 us; one batch
// per thread 18 us more; a test that skips the four divisions of batches within
// one tile 3 us more).
template <class V>
__global__ void k_tile_bounds(const int64_t *__restrict__ off, int64_t n_batch, int64_t n_req, int64_t n_tiles,
                              uint64_t magic, V *__restrict__ part, const TileQueue q, int64_t most, int *status) {
  let_next();
  int bad = 0;
  const int lane = threadIdx.x & 31;
  const int64_t stride = 4 * (int64_t)gridDim.x * blockDim.x;
  // a warp's lanes stay together, for queue_add
  for (int64_t w0 = 4 * (blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u)); w0 <= n_batch; w0 += stride) {
    const int64_t b0 = w0 + 4 * lane;
    int64_t v[5];  // the offsets of batches b0 - 1 .. b0 + 3
    v[0] = b0 > 0 && b0 <= n_batch ? __ldg(off + b0 - 1) : 0;
    if (b0 + 3 <= n_batch) {
      const longlong2 x = __ldg(reinterpret_cast<const longlong2 *>(off + b0)),
                      y = __ldg(reinterpret_cast<const longlong2 *>(off + b0 + 2));
      v[1] = x.x;
      v[2] = x.y;
      v[3] = y.x;
      v[4] = y.y;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k + 1] = b0 + k <= n_batch ? __ldg(off + b0 + k) : n_req;
    }
    if (b0 == 0 && v[1] != 0) bad = 1;
    int64_t c = clampi(v[0], 0, n_req);
    int64_t t0 = b0 > 0 ? div_magic(kTW * (b0 - 1) + c, magic) : -1;
    uint32_t big[kQClasses] = {};  // bit k: batch b0 - 1 + k
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t b = b0 + k;
      if (b > n_batch) break;
      if (b > 0 && v[k] > v[k + 1]) bad = 1;
      const int64_t cb = clampi(v[k + 1], 0, n_req), n = cb - c;
      if (b > 0 && n > most) big[0] |= 1u << k;
      if (b > 0 && n > most && n > kQWarp) big[1] |= 1u << k;
      if (b > 0 && n > most && n > kQTeam) big[2] |= 1u << k;
      const int64_t tb = div_magic(kTW * b + cb, magic);
      if (b == n_batch && v[k + 1] != n_req) bad = 1;
      const int64_t tmax = b == n_batch ? n_tiles : min(tb, n_tiles);
      for (int64_t t = t0 + 1; t <= tmax; ++t) part[t] = (V)b;
      t0 = tb;
      c = cb;
    }
    if (__any_sync(kFull, big[0] != 0u)) {
#pragma unroll
      for (int k = 0; k < kQClasses; ++k)
        queue_add<V>(q, k, big[k] & ~(k + 1 < kQClasses ? big[k + 1 < kQClasses ? k + 1 : 0] : 0u), b0 - 1, lane);
    }
  }
  if (bad) flag(status, kStatusData);
}

// Entry i of the queue.
__device__ __forceinline__ int64_t queued_batch(const TileArgs &a, int64_t i) {
  const int64_t b = a.bound32 ? (int64_t)static_cast<const uint32_t *>(a.queue.list)[i]
                              : static_cast<const int64_t *>(a.queue.list)[i];
  return clampi(b, 0, a.n_batch - 1);
}

__device__ __forceinline__ int64_t tile_bound(const TileArgs &a, int64_t t) {
  return a.bound32 ? (int64_t)a.bound32[t] : a.bound[t];
}

// The smallest m in [lo, hi] for which at(m) holds (hi where none does), for
// two searches by a warp at once: lanes 0..15 make the first, the others the
// second.  16 values are looked at per round and search.
template <class F>
__device__ __forceinline__ int64_t half_warp_search(int lane, int64_t lo, int64_t hi, F &&at) {
  const int half = lane >> 4, l = lane & 15;
  while (__any_sync(kFull, lo < hi)) {
    const int64_t m = lo + (((hi - lo) * l) >> 4);
    const bool in = lo >= hi || at(m);
    const uint32_t bal = (__ballot_sync(kFull, in) >> (16 * half)) & 0xffffu;
    const int c = bal ? __ffs(bal) - 1 : 16;  // the first c probes lie before the result
    const int64_t before = __shfl_sync(kFull, m, 16 * half + max(c - 1, 0)),
                  after = __shfl_sync(kFull, m, 16 * half + min(c, 15));
    if (lo < hi) {
      if (c < 16) hi = after;
      lo = c > 0 ? before + 1 : hi;
    }
  }
  return lo;
}

// The bounds of tile t by a warp's own search, for inputs of at most one tile
// per warp: 20,000 batches take four rounds of one load each, less than
// k_tile_bounds and the gap after it.
__device__ __forceinline__ void tile_search(const TileArgs &a, int64_t t, int lane, int64_t *b0, int64_t *b1) {
  const int64_t tile = t + (lane >> 4), target = tile * a.D;
  const int64_t b = half_warp_search(lane, tile < a.n_tiles ? 0 : a.n_batch, a.n_batch, [&](int64_t m) {
    return kTW * m + clampi(a.off[m], 0, a.n_req) >= target;
  });  // tile n_tiles ends at n_batch
  *b0 = __shfl_sync(kFull, b, 0);
  *b1 = __shfl_sync(kFull, b, 16);
}

// ---------------------------------------------------------------- loads

struct Quad {
  int4 p, c, x;  // x: phases (step 1) or tenants (step 3)
};

// A tile's request arrays from its first staged request (16-byte aligned);
// lim: requests from there to the end of the arrays.
struct TileSrc {
  const int32_t *p, *c, *ph, *u;
  int lim;
};

// Four requests from index e (a multiple of 4).  Past the end of the arrays: the
// last request again, which no sum or share of the tile takes.
template <bool X>
__device__ __forceinline__ Quad load_quad(const int32_t *p, const int32_t *c, const int32_t *x, int e, int lim) {
  Quad q;
  if (e + 4 <= lim) {
    q.p = *reinterpret_cast<const int4 *>(p + e);
    q.c = *reinterpret_cast<const int4 *>(c + e);
    q.x = X ? *reinterpret_cast<const int4 *>(x + e) : make_int4(0, 0, 0, 0);
  } else {
    q.p = q.c = q.x = make_int4(0, 0, 0, 0);
    if (e < lim) {
      const int i1 = min(e + 1, lim - 1), i2 = min(e + 2, lim - 1);
      q.p = make_int4(p[e], p[i1], p[i2], p[i2]);
      q.c = make_int4(c[e], c[i1], c[i2], c[i2]);
      if (X) q.x = make_int4(x[e], x[i1], x[i2], x[i2]);
    }
  }
  return q;
}

// ---------------------------------------------------------------- step 1: prefixes

struct Req8 {
  Quad q[2];
};

__device__ __forceinline__ Req8 load_req8(const TileSrc &t, int e) {
  Req8 r;
  r.q[0] = load_quad<true>(t.p, t.c, t.ph, e, t.lim);
  r.q[1] = load_quad<true>(t.p, t.c, t.ph, e + 4, t.lim);
  return r;
}

// Sums of 8 requests whose p and c are below kTSmall: S1, S2, S3 + prefills << 55.
struct TSum {
  uint32_t s1, s2;
  uint64_t s3;
};

// The first `take` of 8 requests.
__device__ __forceinline__ TSum sum_req8(const Req8 &r, int take) {
  TSum s{0u, 0u, 0ull};
  uint32_t f = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const Quad &v = r.q[h];
    const int32_t p[4] = {v.p.x, v.p.y, v.p.z, v.p.w}, c[4] = {v.c.x, v.c.y, v.c.z, v.c.w},
                  q[4] = {v.x.x, v.x.y, v.x.z, v.x.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = 4 * h + k < take;
      const uint32_t pk = in ? (uint32_t)p[k] : 0u;
      s.s1 += pk;
      s.s2 += in ? (uint32_t)c[k] : 0u;
      s.s3 += (uint64_t)pk * pk;
      f += in ? (uint32_t)q[k] : 0u;
    }
  }
  s.s3 += (uint64_t)f << 55;
  return s;
}

// Prefixes of the tile's requests; true when some p or c is too large for
// them (or negative) or some phase is not 0 or 1.
template <int MODE>
__device__ __forceinline__ bool tile_prefix(WarpTile<MODE> &wt, const TileSrc &src, int cnt, int lane) {
  uint32_t big = 0;
  int e = 8 * lane;
  Req8 nx = load_req8(src, e);
#pragma unroll 1
  for (int k = 0; k * 256 <= cnt; ++k) {
    const Req8 r = nx;
    e += 256;
    if (k * 256 + 256 <= cnt) nx = load_req8(src, e);
    const Quad &x = r.q[0], &y = r.q[1];
    const uint32_t op = (uint32_t)(x.p.x | x.p.y | x.p.z | x.p.w | y.p.x | y.p.y | y.p.z | y.p.w | x.c.x | x.c.y |
                                   x.c.z | x.c.w | y.c.x | y.c.y | y.c.z | y.c.w);
    const uint32_t of = (uint32_t)(x.x.x | x.x.y | x.x.z | x.x.w | y.x.x | y.x.y | y.x.z | y.x.w);
    big |= (op & ~(kTSmall - 1u)) | (of & ~1u);
    TSum s = sum_req8(r, 8);
    const TSum o = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t x1 = __shfl_up_sync(kFull, s.s1, d), x2 = __shfl_up_sync(kFull, s.s2, d);
      const uint64_t x3 = __shfl_up_sync(kFull, s.s3, d);
      if (lane >= d) {
        s.s1 += x1;
        s.s2 += x2;
        s.s3 += x3;
      }
    }
    if (lane == 31) wt.tot[k] = make_uint4(s.s1, s.s2, (uint32_t)s.s3, (uint32_t)(s.s3 >> 32));
    s.s3 -= o.s3;
    wt.pre[32 * k + lane] = make_uint4(s.s1 - o.s1, s.s2 - o.s2, (uint32_t)s.s3, (uint32_t)(s.s3 >> 32));
  }
  return __any_sync(kFull, big != 0u);
}

// Sums of the requests before index x of its 256.
template <int MODE>
__device__ __forceinline__ TSum prefix_at(const WarpTile<MODE> &wt, const TileSrc &src, int x) {
  const uint4 v = wt.pre[x >> 3];
  TSum r{v.x, v.y, (uint64_t)v.z | ((uint64_t)v.w << 32)};
  if (x & 7) {
    const TSum s = sum_req8(load_req8(src, x & ~7), x & 7);
    r.s1 += s.s1;
    r.s2 += s.s2;
    r.s3 += s.s3;
  }
  return r;
}

// ---------------------------------------------------------------- step 2: batches

// Share constants of a batch of n requests in segment s; kTab: n is within the
// K table (every staged batch).
template <int MODE, bool kTab>
__device__ __forceinline__ TileRec tile_record(const TileArgs &a, const TSmem<MODE> &ts, int s, int64_t n) {
  TileRec r;
  if (MODE & M_F32) {
    const float *k = ts.cf[s];
    const float fn = (float)n;
    r.k = make_uint4(__float_as_uint(__fadd_rn(__fdiv_rn(k[0], fn), __fmul_rn(k[4], fn))), __float_as_uint(k[1]),
                     __float_as_uint(k[2]), __float_as_uint(k[3]));
    r.a = make_uint4(0u, 0u, 0u, 0u);
    return r;
  }
  bool slow = false;
  const SegS &sg = ts.seg[s];
  i128 kf;
  if ((MODE & M_FIX) && kTab) {
    kf = a.mp.ktab[s * (kTabN + 1) + (int)n].kf;
    slow = kf.hi == kKSlowHi;
  } else {
    kf = batch_const_w<MODE>(a, s, n, &slow);
  }
  const i128 k = (MODE & M_FIX) ? add128(kf, sg.A13) : kf;
  // fast: 2^64 <= constant < 2^95 (then the share, below 2^95 more, is in [2^64, 2^96)) and A2 < 2^64
  const bool fast = (MODE & M_FIX) && !slow && sg.a2_narrow && k.hi != 0 && k.hi < (1ull << 31);
  r.k = make_uint4((uint32_t)k.lo, (uint32_t)(k.lo >> 32), (uint32_t)k.hi, (uint32_t)(sg.E + 32) << 20);
  r.a = make_uint4((uint32_t)sg.A2.lo, (uint32_t)(sg.A2.lo >> 32),
                   ((uint32_t)n << 4) | (fast ? 8u : 0u) | (slow ? 4u : 0u) | (uint32_t)s, (uint32_t)(k.hi >> 32));
  return r;
}

// A batch's outputs.
template <int MODE>
__device__ __forceinline__ void tile_emit(const TileArgs &a, const TSmem<MODE> &ts, int64_t b, const BatchAgg &g,
                                          int s) {
  if ((MODE & M_ATTR) && (MODE & M_F32)) {
    if (a.T32) {
      const float *k = ts.cf[s];
      float T = __fmaf_rn(k[1], (float)g.s1, k[0]);
      T = __fmaf_rn(k[2], (float)g.s2, T);
      T = __fmaf_rn(k[3], (float)g.s3, T);
      T = __fmaf_rn(k[4], (float)(g.n * g.n), T);
      a.T32[b] = g.n > 0 ? T : 0.0f;
    }
  } else if ((MODE & M_ATTR) && (MODE & M_FIX)) {
    if (a.T) a.T[b] = eq1_exact(a.mp, ts.fx[s], ts.seg[s].t32, s, g);
  } else if (MODE & M_FIT) {
    const int64_t i = b - a.f_lo;
    a.bfeat[i] = g.s1;
    a.bfeat[a.f_stride + i] = g.s2;
    a.bfeat[2 * a.f_stride + i] = g.s3;
    a.bfeat[3 * a.f_stride + i] = g.n;
    a.bseg[i] = g.n > 0 ? (uint8_t)s : (uint8_t)255;
  } else {
    emit_batch<MODE>(a, b, g, s, nullptr);
  }
}

// ---------------------------------------------------------------- step 3: requests

// The CTA's tenant table, which follows TSmem (formed again in the functions
// kept out of line, so that the loops hold it in fewer registers).
template <int MODE>
__device__ __forceinline__ TenTab tile_table(const TileArgs &a, const TSmem<MODE> &ts) {
  return ten_table(reinterpret_cast<const uint32_t *>(&ts + 1), kHotMax, a.H, a.n_tenants, a.ten_pend);
}

// The general path of one request.  Out of line: the fast path leaves it the
// rare ones (fp64 mode, values out of range).
template <int MODE>
__device__ __noinline__ void tile_slow(const TileArgs &a, const TSmem<MODE> &ts, const TileRec &rec, int64_t n,
                                       int64_t i, int32_t p, int32_t c, int32_t u) {
  const int s = (int)(rec.a.z & 3u);
  const bool slow = (rec.a.z & 4u) != 0u;
  const SegS &sg = ts.seg[s];
  i128 kf = mk128((uint64_t)rec.k.x | ((uint64_t)rec.k.y << 32), (uint64_t)rec.k.z | ((uint64_t)rec.a.w << 32));
  if (MODE & M_FIX) kf = add128(kf, neg128(sg.A13));
  p = max(p, 0);
  c = max(c, 0);
  const Rounded r = (MODE & M_FIX) && !slow && p <= kPMaxFix
                        ? share_fix(sg, kf, (uint32_t)p, (uint32_t)c)
                        : share_slow(a.mp, s, (MODE & M_FIX) != 0, kf, p, c, n);
  if (a.share) __stcs(a.share + i, r.d);
  if (MODE & M_TEN) {
    int bad = 0;
    tenant_add_any(tile_table(a, ts), u, r, &bad);
    if (bad) flag(a.status, kStatusData);
  }
}

// Constant + A2 c on the fast path: below 2^96, no carry leaves word 2.
__device__ __forceinline__ double tile_value(const TileRec &r, uint32_t k0, uint32_t k1, uint32_t k2, int32_t c) {
  uint32_t v0, v1, v2;
  asm("mad.lo.cc.u32 %0, %3, %5, %6;\n\t"
      "madc.hi.cc.u32 %1, %3, %5, %7;\n\t"
      "addc.u32 %2, %8, 0;\n\t"
      "mad.lo.cc.u32 %1, %4, %5, %1;\n\t"
      "madc.hi.u32 %2, %4, %5, %2;"
      : "=&r"(v0), "=&r"(v1), "=&r"(v2)
      : "r"(r.a.x), "r"(r.a.y), "r"((uint32_t)c), "r"(k0), "r"(k1), "r"(k2));
  return round_top(v0, v1, v2, r.k.w);
}

// A request's exact share on the fast path, rounded to nearest even; false
// where the path does not apply.  The constant is K + A1 + A3 for p = 1; a
// prefill adds (p - 1)(A1 + A3 (p + 1)).  With p_narrow (A1 < 2^95, A3 < 2^64)
// and p <= 2^24 that is below 2^120, so the 128-bit sum is exact; it must be
// below 2^95.
__device__ __forceinline__ bool tile_share(const SegS *segs, const TileRec &r, int32_t p, int32_t c, double *d) {
  uint32_t k0 = r.k.x, k1 = r.k.y, k2 = r.k.z;
  bool ok = (r.a.z & 8u) != 0u;
  if (p != 1) {
    const SegS &sg = segs[r.a.z & 3u];
    ok = ok && p > 1 && p <= kPMaxFix && sg.p_narrow;
    const i128 g = add128(sg.A1, mul_u64_u32(sg.A3.lo, (uint32_t)p + 1u));
    const i128 b = add128(mk128((uint64_t)k0 | ((uint64_t)k1 << 32), (uint64_t)k2), mul128_u32(g, (uint32_t)p - 1u));
    k0 = (uint32_t)b.lo;
    k1 = (uint32_t)(b.lo >> 32);
    k2 = (uint32_t)b.hi;
    ok = ok && b.hi < (1ull << 31);
  }
  *d = tile_value(r, k0, k1, k2, max(c, 0));
  return ok;
}

__device__ __forceinline__ void store4(double *p, const double *d) {
  asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(d[0]), "d"(d[1]), "d"(d[2]), "d"(d[3])
               : "memory");
}

// One request through the fast path where it applies, else the general one.
template <int MODE>
__device__ __forceinline__ bool tile_one(const TileArgs &a, const TenTab &tt, const TSmem<MODE> &ts, const TileRec &rec,
                                         int64_t n, int64_t i, int32_t p, int32_t c, int32_t u, double *d) {
  bool ok = (MODE & M_FIX) && tile_share(ts.seg, rec, p, c, d);
  if (MODE & M_TEN)
    ok = ok && tenant_add_pos(tt, (uint32_t)u, (uint32_t)__double2loint(*d), (uint32_t)__double2hiint(*d));
  if (!ok) tile_slow<MODE>(a, ts, rec, n, i, p, c, u);
  return ok;
}

// One request of the fp32 variant.
template <int MODE>
__device__ __forceinline__ float tile_one_f32(const TileArgs &a, const TenTab &tt, const TileRec &rec, int32_t p,
                                              int32_t c, int32_t u, int *bad) {
  const Share32 q{__uint_as_float(rec.k.x), __uint_as_float(rec.k.y), __uint_as_float(rec.k.z),
                  __uint_as_float(rec.k.w)};
  const float s = share_f32(q, p, c);
  if (MODE & M_TEN) {
    // a positive normal float's double: the same significand, the exponent rebiased
    const uint32_t f = __float_as_uint(s);
    const bool normal = f >= 0x00800000u && f < 0x7f800000u;
    if (!normal || !tenant_add_pos(tt, (uint32_t)u, f << 29, (f >> 3) + ((1023u - 127u) << 20)))
      tenant_add_any(tt, u, decompose((double)s), bad);
  }
  return s;
}

// The record of the request at index e; before the tile's first batch, the first.
template <int MODE>
__device__ __forceinline__ int tile_rank(const WarpTile<MODE> &wt, int e) {
  const int r = (int)wt.rank[e >> 5] + __popc(wt.bits[e >> 5] & ((2u << (e & 31)) - 1u));
  return max(min(r, Geo<MODE>::kRec) - 1, 0);
}

// The tile's n listed requests, one per lane: prefills, tenants and values off
// the common path, with every lane busy.
template <int MODE, bool kWalk>
__device__ __forceinline__ void tile_rest(const TileArgs &a, const TenTab &tt, const TSmem<MODE> &ts,
                                          const WarpTile<MODE> &wt, const TileSrc &src, int64_t rbase, int n,
                                          int64_t n_walk, int lane) {
  __syncwarp();
  int bad = 0;
#pragma unroll 1
  for (int k = lane; k < n; k += 32) {
    const int e = wt.list[k];
    const TileRec &rec = wt.rec[tile_rank(wt, e)];
    const int32_t p = src.p[e], c = src.c[e], u = (MODE & M_TEN) ? src.u[e] : 0;
    if (MODE & M_F32) {
      const float f = tile_one_f32<MODE>(a, tt, rec, kWalk ? max(p, 0) : p, kWalk ? max(c, 0) : c, u, &bad);
      if (a.share32) __stcs(a.share32 + rbase + e, f);
    } else {
      double d;
      if (tile_one<MODE>(a, tt, ts, rec, kWalk ? n_walk : (int64_t)(rec.a.z >> 4), rbase + e, p, c, u, &d) && a.share)
        __stcs(a.share + rbase + e, d);
    }
  }
  if (bad) flag(a.status, kStatusData);
}

// The tile's shares, four consecutive requests per lane and step.  The loop
// takes decode requests (p = 1; fp32 variant: any) on the common path, without a
// call; the rest goes to the warp's list, worked off after it.  A lane loads
// another record where a batch starts among its four (leaving what lies past
// the start to the list, where batches average 40 requests and more, was
// no faster: 1.36e8 requests of batches of 16 to 256, 840 us either way, and the
// second copy of the loop cost the fp32 variant 3 %).  vec: the share array allows
// 32-byte (fp32: 16-byte) stores.  kWalk: a part of a batch of n_walk requests on its own, whose values may
// be negative (walk_batch).
template <int MODE, bool kWalk>
__device__ __forceinline__ void tile_shares(const TileArgs &a, const TenTab &tt, const TSmem<MODE> &ts,
                                            WarpTile<MODE> &wt, const TileSrc &src, int64_t rbase, int first, int cnt,
                                            bool vec, int64_t n_walk, int lane) {
  constexpr bool kTen = (MODE & M_TEN) != 0, kF32 = (MODE & M_F32) != 0;
  if (!(MODE & (M_FIX | M_F32))) {
    // fp64 mode has no common path: one request per lane, in order
    for (int e = lane; e < cnt; e += 32) {
      if (e < first) continue;
      const TileRec &rec = wt.rec[tile_rank(wt, e)];
      tile_slow<MODE>(a, ts, rec, kWalk ? n_walk : (int64_t)(rec.a.z >> 4), rbase + e, src.p[e], src.c[e],
                      kTen ? src.u[e] : 0);
    }
    return;
  }
  Quad nx = load_quad<kTen>(src.p, src.c, src.u, 4 * lane, src.lim);
#pragma unroll 1
  for (int b = 0; b < cnt; b += 128) {
    const int e = b + 4 * lane;
    const Quad v = nx;
    if (b + 128 < cnt) nx = load_quad<kTen>(src.p, src.c, src.u, e + 128, src.lim);
    int32_t p[4] = {v.p.x, v.p.y, v.p.z, v.p.w}, c[4] = {v.c.x, v.c.y, v.c.z, v.c.w};
    if (kWalk) {
#pragma unroll
      for (int k = 0; k < 4; ++k) p[k] = max(p[k], 0), c[k] = max(c[k], 0);
    }
    const uint32_t u[4] = {(uint32_t)v.x.x, (uint32_t)v.x.y, (uint32_t)v.x.z, (uint32_t)v.x.w};
    // the quad's requests that are the tile's
    const int hi = min(max(cnt - e, 0), 4), lo = max(first - e, 0);
    const uint32_t vm = ((1u << hi) - 1u) & (15u << lo);
    const uint32_t word = wt.bits[b / 32 + (lane >> 3)];
    const int sh = e & 31;
    const uint32_t hb = (word >> sh) & 14u;
    // record of the first request; -1 before the tile's first batch
    const int r0 = min((int)wt.rank[b / 32 + (lane >> 3)] + __popc(word & ((2u << sh) - 1u)), Geo<MODE>::kRec - 4) - 1;
    TileRec rec = wt.rec[max(r0, 0)];
    bool go[4];
    uint32_t dlo[4], dhi[4];
    float f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k > 0 && ((hb >> k) & 1u)) rec = wt.rec[max(r0 + __popc(hb & ((2u << k) - 1u)), 0)];
      go[k] = ((vm >> k) & 1u) != 0u;
      if (kF32) {
        const Share32 q{__uint_as_float(rec.k.x), __uint_as_float(rec.k.y), __uint_as_float(rec.k.z),
                        __uint_as_float(rec.k.w)};
        f[k] = share_f32(q, p[k], c[k]);
        // a positive normal float's double: the same significand, the exponent rebiased
        const uint32_t x = __float_as_uint(f[k]);
        dlo[k] = x << 29;
        dhi[k] = (x >> 3) + ((1023u - 127u) << 20);
        if (kTen) go[k] = go[k] && x - 0x00800000u < 0x7f000000u;
      } else {
        go[k] = go[k] && (MODE & M_FIX) && (rec.a.z & 8u) && p[k] == 1;
        const double d = tile_value(rec, rec.k.x, rec.k.y, rec.k.z, c[k]);
        dlo[k] = (uint32_t)__double2loint(d);
        dhi[k] = (uint32_t)__double2hiint(d);
      }
    }
    if (kTen) ten_add4(tt, go, u, dlo, dhi);
    uint32_t dm = vm;
#pragma unroll
    for (int k = 0; k < 4; ++k) dm &= go[k] ? ~(1u << k) : ~0u;
    const int64_t i0 = rbase + e;
    if (kF32 && a.share32) {
      if (vec && (go[0] && go[1] && go[2] && go[3])) {
        __stcs(reinterpret_cast<float4 *>(a.share32 + i0), make_float4(f[0], f[1], f[2], f[3]));
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (go[k]) __stcs(a.share32 + i0 + k, f[k]);
      }
    }
    if (!kF32 && a.share) {
      double d[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) d[k] = __hiloint2double((int)dhi[k], (int)dlo[k]);
      if (vec && (go[0] && go[1] && go[2] && go[3])) {
        store4(a.share + i0, d);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (go[k]) __stcs(a.share + i0 + k, d[k]);
      }
    }
    if (dm) {
      // slots by a shared-memory add: few lanes come here, and the list's order is free
      uint32_t at = atomicAdd(&wt.n_list, (uint32_t)__popc(dm));
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if ((dm >> k) & 1u) wt.list[at++] = (uint16_t)(e + k);
    }
  }
  __syncwarp();
  const int nl = (int)wt.n_list;
  if (nl > 0) tile_rest<MODE, kWalk>(a, tt, ts, wt, src, rbase, nl, n_walk, lane);
}

// One batch walked by a warp from global memory: sums, then a strided share pass.
// (Out of line and without tile_shares' loop: a call that needs more registers
// costs the tiles' loop some.)
template <int MODE>
__device__ __noinline__ void walk_alone(const TileArgs &a, TSmem<MODE> &ts, int64_t b, int64_t r0, int64_t n) {
  const TenTab tt = tile_table(a, ts);
  constexpr int kThreads = 32;
  const int tid = (int)(threadIdx.x & 31);
  int bad = 0;
  Sums acc{0, 0, 0, 0};
  for (int64_t i = tid; i < n; i += 4 * kThreads) {
    int32_t p[4], c[4], f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t j = i + k * kThreads;
      p[k] = j < n ? a.p[r0 + j] : 0;
      c[k] = j < n ? a.c[r0 + j] : 0;
      f[k] = j < n ? a.ph[r0 + j] : 0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      check_req(p[k], c[k], f[k], &bad);
      acc.s1 += p[k];
      acc.s2 += c[k];
      acc.s3 += (int64_t)p[k] * p[k];
      acc.ph |= f[k];
    }
  }
  acc = warp_sum(acc);
  const BatchAgg g{acc.s1, acc.s2, acc.s3, n, acc.ph > 0};
  const int s = segment_of(a.mp, g);
  if (tid == 0) tile_emit<MODE>(a, ts, b, g, s);
  if ((MODE & M_ATTR) && n > 0) {
    const TileRec rec = tile_record<MODE, false>(a, ts, s, n);
    for (int64_t i = tid; i < n; i += kThreads) {
      const int64_t q = r0 + i;
      const int32_t p = a.p[q], c = a.c[q], u = (MODE & M_TEN) ? a.ten[q] : 0;
      if (MODE & M_F32) {
        const float f = tile_one_f32<MODE>(a, tt, rec, max(p, 0), max(c, 0), u, &bad);
        if (a.share32) __stcs(a.share32 + q, f);
      } else {
        double d;
        if (tile_one<MODE>(a, tt, ts, rec, n, q, p, c, u, &d) && a.share) __stcs(a.share + q, d);
      }
    }
  }
  if (bad) flag(a.status, kStatusData);
}

// A barrier of `kThreads` consecutive threads of the CTA (all of it, or a team).
template <int kThreads>
__device__ __forceinline__ void sync_team() {
  if (kThreads == kTThreads) {
    __syncthreads();
  } else {
    __syncwarp();  // the barrier counts whole warps
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / kThreads), "n"(kThreads) : "memory");
  }
}

// One batch walked by `kThreads` threads (a warp, a team, or the CTA) from global
// memory: sums, then its shares in parts, each as a tile of one batch that a
// warp attributes in its own tile's memory.
template <int MODE, int kThreads>
__device__ __noinline__ void walk_batch(const TileArgs &a, TSmem<MODE> &ts, int64_t b, int64_t r0, int64_t n) {
  constexpr int kWarps = kThreads / 32;
  const int tid = (int)threadIdx.x % kThreads, lane = tid & 31;
  const int64_t rbase = r0 & ~(int64_t)3, end = r0 + n;
  int bad = 0;
  Sums acc{0, 0, 0, 0};
  for (int64_t q0 = rbase + 4 * tid; q0 < end; q0 += 8 * kThreads) {
    Quad v[2];  // both quads' loads in flight
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t q = q0 + 4 * kThreads * h, left = a.n_req - q;
      v[h].p = v[h].c = v[h].x = make_int4(0, 0, 0, 0);
      if (q < end) v[h] = load_quad<true>(a.p + q, a.c + q, a.ph + q, 0, left < 4 ? (int)left : 4);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t q = q0 + 4 * kThreads * h;
      int32_t p[4] = {v[h].p.x, v[h].p.y, v[h].p.z, v[h].p.w}, c[4] = {v[h].c.x, v[h].c.y, v[h].c.z, v[h].c.w},
              f[4] = {v[h].x.x, v[h].x.y, v[h].x.z, v[h].x.w};
      if (q < r0 || q + 4 > end) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (q + k < r0 || q + k >= end) p[k] = c[k] = f[k] = 0;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        check_req(p[k], c[k], f[k], &bad);
        acc.s1 += p[k];
        acc.s2 += c[k];
        acc.s3 += (int64_t)p[k] * p[k];
        acc.ph |= f[k];
      }
    }
  }
  acc = warp_sum(acc);
  if (kWarps > 1) {
    const Sums *red = ts.red + threadIdx.x / kThreads * kWarps;
    if (lane == 0) ts.red[threadIdx.x >> 5] = acc;
    sync_team<kThreads>();
    acc = Sums{0, 0, 0, 0};
#pragma unroll
    for (int w = 0; w < kWarps; ++w) acc = add_sums(acc, red[w]);
    sync_team<kThreads>();  // ts.red is rewritten for the next batch
  }
  const BatchAgg g{acc.s1, acc.s2, acc.s3, n, acc.ph > 0};
  const int s = segment_of(a.mp, g);
  if (tid == 0) tile_emit<MODE>(a, ts, b, g, s);
  if ((MODE & M_ATTR) && n > 0 && ((MODE & M_TEN) || a.share || a.share32)) {
    // parts of whole rows of 128 requests, as many for every warp
    const int64_t rows = (end - rbase + 127) >> 7, most = kWarps * (Geo<MODE>::kCap / 128),
                  parts = kWarps * ((rows + most - 1) / most);
    const int part = 128 * (int)((rows + parts - 1) / parts);
    WarpTile<MODE> &wt = ts.tile[threadIdx.x >> 5];
    for (int i = lane; i <= part / 32 && i < Geo<MODE>::kWords; i += 32) {
      wt.bits[i] = 0;
      wt.rank[i] = 1;
    }
    if (lane == 0) wt.rec[0] = tile_record<MODE, false>(a, ts, s, n);
    const bool vec = (MODE & M_F32) ? ((uintptr_t)a.share32 & 15) == 0 : ((uintptr_t)a.share & 31) == 0;
    const TenTab tt = tile_table(a, ts);
    for (int64_t q = rbase + (int64_t)(tid >> 5) * part; q < end; q += (int64_t)kWarps * part) {
      __syncwarp();
      if (lane == 0) wt.n_list = 0;
      __syncwarp();
      const TileSrc src{a.p + q, a.c + q, a.ph + q, (MODE & M_TEN) ? a.ten + q : nullptr,
                        (int)(a.n_req - q < 0x40000000 ? a.n_req - q : 0x40000000)};
      tile_shares<MODE, true>(a, tt, ts, wt, src, q, q < r0 ? (int)(r0 - q) : 0,
                              end - q < part ? (int)(end - q) : part, vec, n, lane);
    }
    __syncwarp();
  }
  if (bad) flag(a.status, kStatusData);
}

__device__ __forceinline__ void batch_range(const TileArgs &a, int64_t b, int64_t *r0, int64_t *n) {
  *r0 = clampi(a.off[b], 0, a.n_req);
  *n = clampi(a.off[b + 1], *r0, a.n_req) - *r0;
}

// The CTA's list, each of its warps, its teams or all of it taking one batch at a time.
template <int MODE, int kThreads>
__device__ __forceinline__ void walk_list(const TileArgs &a, TSmem<MODE> &ts, int nbig) {
  for (int k = (int)threadIdx.x / kThreads; k < nbig; k += kTThreads / kThreads) {
    int64_t r0, n;
    batch_range(a, ts.big[k], &r0, &n);
    walk_batch<MODE, kThreads>(a, ts, ts.big[k], r0, n);
  }
}

// One class of the queue, each team or CTA taking one batch at a time.
template <int MODE, int kThreads>
__device__ __forceinline__ void walk_class(const TileArgs &a, TSmem<MODE> &ts, int cls, int64_t count) {
  int64_t *turn = ts.big + 3 * ((int)threadIdx.x / kThreads);  // batch, first request, requests
  for (;;) {
    if ((int)threadIdx.x % kThreads == 0) {
      const int64_t i = atomicAdd(a.queue.ctr + kQTaken + cls, 1u);
      turn[0] = -1;
      if (i < count) {
        turn[0] = queued_batch(a, a.queue.at[cls] + i);
        batch_range(a, turn[0], turn + 1, turn + 2);
      }
    }
    sync_team<kThreads>();
    if (turn[0] < 0) break;
    walk_batch<MODE, kThreads>(a, ts, turn[0], turn[1], turn[2]);  // synchronises the team after reading these
  }
  __syncthreads();
}

// The same, each warp one batch at a time, taken one ahead.
template <int MODE>
__device__ __forceinline__ void walk_class_warps(const TileArgs &a, TSmem<MODE> &ts, int cls, int64_t count) {
  const int lane = threadIdx.x & 31;
  unsigned nx = 0;
  if (lane == 0) nx = atomicAdd(a.queue.ctr + kQTaken + cls, 1u);
  for (;;) {
    const int64_t i = __shfl_sync(kFull, nx, 0);
    if (i >= count) break;
    if (lane == 0) nx = atomicAdd(a.queue.ctr + kQTaken + cls, 1u);
    int64_t r0, n;
    const int64_t b = queued_batch(a, a.queue.at[cls] + i);
    batch_range(a, b, &r0, &n);
    walk_batch<MODE, 32>(a, ts, b, r0, n);
  }
  __syncthreads();
}

// The queued batches, the largest class first.  A warp walks a batch with the
// fewest instructions but takes longest for one, a CTA the other way round: so a
// CTA takes large ones and those of a class with few, a team of four warps those
// of a class with two or more for every CTA, a warp the smallest where there are
// half as many again as warps.  Measured on both sides of each line (fp64 shares,
// 256 tenants; 5e7 requests unless said):
//   1,600 a batch, by warps    401 us, teams 612         20,000, by teams 439, CTAs 508
//   4,096 a batch, by warps    407 us, teams 429         30,000, by CTAs  461, teams 488
//   6,000 of 4,000, by warps   223 us, teams 251         60,000, by CTAs  472, teams 614
//   3,100 of 4,000, by teams   162 us, warps 205         500 of 10,000, by teams 105, CTAs 119
// Before the queue, with the CTA whose tile held a batch's start walking it one
// request per thread and turn, 4,096 a batch took 1,307 us, 9,976 930 (415 now),
// 200,000 1,280 (465).  The last CTA out leaves the counters at zero for the next
// call.
template <int MODE>
__device__ __noinline__ void walk_queue(const TileArgs &a, TSmem<MODE> &ts) {
  __syncthreads();  // the list's memory is free
#pragma unroll 1
  for (int c = kQClasses - 1; c >= 0; --c) {
    const int64_t count = min((int64_t)ts.queued[c], a.queue.at[c + 1] - a.queue.at[c]);
    if (c == 0 && 2 * count >= 3 * (int64_t)gridDim.x * kTWarps)
      walk_class_warps<MODE>(a, ts, c, count);
    else if (c <= 1 && count >= 2 * (int64_t)gridDim.x)
      walk_class<MODE, kTTeam>(a, ts, c, count);
    else if (count > 0)
      walk_class<MODE, kTThreads>(a, ts, c, count);
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(a.queue.ctr + kQDone, 1u) == gridDim.x - 1) {
#pragma unroll
      for (int k = 0; k < kQueueWords; ++k) a.queue.ctr[k] = 0u;
    }
  }
}

// ---------------------------------------------------------------- kernel

template <int MODE>
__global__ void __launch_bounds__(kTThreads, 1) k_tiles(const TileArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  TSmem<MODE> &ts = *reinterpret_cast<TSmem<MODE> *>(smem_raw);
  constexpr bool kTen = (MODE & M_TEN) != 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int bad = 0;

  uint32_t *tw = reinterpret_cast<uint32_t *>(smem_raw + sizeof(TSmem<MODE>));
  TenTab tt{};
  if (kTen) {
    tt = tile_table(a, ts);
    for (int i = tid; i < (int)(ten_table_bytes(kHotMax) / 4); i += kTThreads) tw[i] = 0;
  }
  if (MODE & M_ATTR) {
    init_segs<MODE>(a, ts.seg);
    if (tid < 4) ts.fx[tid] = a.mp.fx[tid];
    if ((MODE & M_F32) && tid < 20) ts.cf[tid / 5][tid % 5] = __double2float_rn(a.mp.coef[tid / 5][tid % 5]);
  }
  if (tid == 0) ts.n_big = 0;
  __syncthreads();
  wait_previous();

  WarpTile<MODE> &wt = ts.tile[wid];
  const bool vec = (MODE & M_F32) ? ((uintptr_t)a.share32 & 15) == 0 : ((uintptr_t)a.share & 31) == 0;
  // tile t's batches [b0, b1) and requests [r0, r1) are fetched while the tile
  // before it is worked on
  const int64_t stride = (int64_t)gridDim.x * kTWarps;
  int64_t t = (int64_t)wid * gridDim.x + blockIdx.x, t_end = a.n_tiles;
  if (a.D) {
    // at most one tile per warp: a CTA takes neighbours, so that batches that reach
    // past their tiles, which it walks afterwards, are spread over the CTAs
    const unsigned n = (unsigned)a.n_tiles;  // at most kTWarps a CTA
    t = n * blockIdx.x / gridDim.x + wid;
    t_end = n * (blockIdx.x + 1) / gridDim.x;
  }
  const bool queued = a.queue.list != nullptr;
  const unsigned in_queue = queued && tid < kQClasses ? __ldcg(a.queue.ctr + kQListed + tid) : 0u;
  int64_t b0 = 0, b1 = 0, r0 = 0, r1 = 0;
  // a fit of many batches: the tiles whose first batch is in the range
  const bool ranged = (MODE & M_FIT) && a.f_range != nullptr;
  if (ranged) {
    const int64_t from = lane < 16 ? a.f_lo : a.f_hi;
    const int64_t x = half_warp_search(lane, 0, a.n_tiles, [&](int64_t m) { return tile_bound(a, m) >= from; });
    const int64_t t_lo = __shfl_sync(kFull, x, 0);
    t_end = __shfl_sync(kFull, x, 16);
    t += t_lo;
    if (blockIdx.x == 0 && tid == 0) {
      a.f_range[0] = clampi(tile_bound(a, t_lo) - a.f_lo, 0, a.f_stride);
      a.f_range[1] = clampi(tile_bound(a, t_end) - a.f_lo, a.f_range[0], a.f_stride);
    }
  }
  if (a.D) {
    // k_tile_bounds' checks of the offsets
    const int64_t threads = (int64_t)gridDim.x * kTThreads;
    for (int64_t i = blockIdx.x * (int64_t)kTThreads + tid; i < a.n_batch; i += threads)
      if (a.off[i] > a.off[i + 1]) bad = 1;
    if (blockIdx.x == 0 && tid == 0 && (a.off[0] != 0 || a.off[a.n_batch] != a.n_req)) bad = 1;
  }
  if (t < t_end) {
    if (a.D) {
      tile_search(a, t, lane, &b0, &b1);
    } else {
      b0 = tile_bound(a, t);
      b1 = tile_bound(a, t + 1);
    }
    b0 = clampi(b0, ranged ? a.f_lo : 0, ranged ? a.f_hi : a.n_batch);
    b1 = clampi(b1, b0, a.n_batch);
    r0 = clampi(a.off[b0], 0, a.n_req);
    r1 = clampi(a.off[b1], r0, a.n_req);
  }
  if (tid < kQClasses) ts.queued[tid] = in_queue;
  while (t < t_end) {
    const int64_t tn = t + stride;
    int64_t n0 = 0, n1 = 0;
    if (tn < t_end) {
      n0 = tile_bound(a, tn);
      n1 = tile_bound(a, tn + 1);
    }
    if (b1 - b0 > Geo<MODE>::kNb) {
      b1 = b0 + Geo<MODE>::kNb;  // invalid offsets
      bad = 1;
    }
    const int nb = (int)(b1 - b0);
    const int64_t rbase = r0 & ~(int64_t)3;
    int64_t off0 = lane <= nb ? a.off[b0 + lane] : 0;  // the first round's offsets
    if (r1 - rbase > Geo<MODE>::kCap) {
      // the last batch reaches too far: the tile's requests end at its start
      r1 = nb > 0 ? clampi(a.off[b1 - 1], r0, a.n_req) : r0;
      if (r1 - rbase > Geo<MODE>::kCap) r1 = rbase + Geo<MODE>::kCap;  // invalid offsets
    }
    const int cnt = (int)(r1 - rbase), first = (int)(r0 - rbase);
    const TileSrc src{a.p + rbase, a.c + rbase, a.ph + rbase, kTen ? a.ten + rbase : nullptr,
                      (int)(a.n_req - rbase < 0x40000000 ? a.n_req - rbase : 0x40000000)};

    // 1. prefixes
    if (MODE & M_ATTR) {
      for (int i = lane; i < Geo<MODE>::kWords; i += 32) {
        wt.bits[i] = 0;
        if (i == 0) {
          wt.rank[0] = 0;
          wt.n_list = 0;
        }
      }
    }
    const bool wide = cnt > first && tile_prefix(wt, src, cnt, lane);
    __syncwarp();
    n0 = clampi(n0, ranged ? a.f_lo : 0, ranged ? a.f_hi : a.n_batch);
    n1 = clampi(n1, n0, a.n_batch);
    int64_t nr0 = a.off[n0], nr1 = a.off[n1];

    // 2. batches
    int before = 0;  // non-empty batches of earlier rounds
    bool direct = false;
#pragma unroll 1
    for (int i0 = 0; i0 < nb; i0 += 31) {
      // lane 31 holds the bound after lane 30's batch
      const int i = i0 + lane;
      const int64_t o0 = i0 == 0 ? off0 : i <= nb ? a.off[b0 + i] : 0;
      const int64_t o1 = __shfl_down_sync(kFull, o0, 1);
      const bool act = lane < 31 && i < nb;
      // staged: both bounds among the tile's requests, in order
      const uint64_t d0 = (uint64_t)(o0 - rbase);
      const int x = d0 <= (uint64_t)cnt ? (int)d0 : -1;
      const int x1 = __shfl_down_sync(kFull, x, 1);
      const bool staged = act && x >= 0 && x1 >= x && !wide;
      TSum lo{0u, 0u, 0ull};
      if (i <= nb && x >= 0) lo = prefix_at(wt, src, x);
      const TSum hi{__shfl_down_sync(kFull, lo.s1, 1), __shfl_down_sync(kFull, lo.s2, 1),
                    __shfl_down_sync(kFull, lo.s3, 1)};
      const int n = staged ? x1 - x : 0;
      const uint32_t ne = __ballot_sync(kFull, n > 0);
      if (staged) {
        constexpr uint64_t kM55 = (1ull << 55) - 1ull;
        int64_t s1 = (int64_t)hi.s1 - lo.s1, s2 = (int64_t)hi.s2 - lo.s2;
        int64_t s3 = (int64_t)(hi.s3 & kM55) - (int64_t)(lo.s3 & kM55);
        int f = (int)(hi.s3 >> 55) - (int)(lo.s3 >> 55);
        for (int k = x >> 8; k < (x1 >> 8); ++k) {
          const uint4 v = wt.tot[k];
          const uint64_t v3 = (uint64_t)v.z | ((uint64_t)v.w << 32);
          s1 += v.x;
          s2 += v.y;
          s3 += (int64_t)(v3 & kM55);
          f += (int)(v3 >> 55);
        }
        const BatchAgg g{s1, s2, s3, n, f > 0};
        const int sg = segment_of(a.mp, g);
        const int rank = before + __popc(ne & ((1u << lane) - 1u));
        if ((MODE & M_ATTR) && n > 0 && rank < Geo<MODE>::kRec) {
          wt.rec[rank] = tile_record<MODE, true>(a, ts, sg, n);
          atomicOr(&wt.bits[x >> 5], 1u << (x & 31));
          for (int w = (x >> 5) + 1; w <= (x1 >> 5); ++w) wt.rank[w] = (uint16_t)(rank + 1);
        }
        tile_emit<MODE>(a, ts, b0 + i, g, sg);
      }
      before += __popc(ne);
      direct |= __any_sync(kFull, act && !staged);
    }
    __syncwarp();
    nr0 = clampi(nr0, 0, a.n_req);
    nr1 = clampi(nr1, nr0, a.n_req);

    // 3. requests
    if ((MODE & M_ATTR) && !wide && (kTen || a.share || a.share32)) {
      tile_shares<MODE, false>(a, tt, ts, wt, src, rbase, first, cnt, vec, 0, lane);
    }
    if (direct) {
      // the last batch; every batch of a wide tile; the queued ones later
      for (int i = 0; i < nb; ++i) {
        const int64_t o0 = a.off[b0 + i], o1 = a.off[b0 + i + 1];
        const uint64_t d0 = (uint64_t)(o0 - rbase), d1 = (uint64_t)(o1 - rbase);
        if (d0 <= d1 && d1 <= (uint64_t)cnt && !wide) continue;
        const int64_t c0 = clampi(o0, 0, a.n_req), c1 = clampi(o1, c0, a.n_req);
        if (c0 != o0 || c1 != o1) bad = 1;
        if (queued && c1 - c0 > Geo<MODE>::kCap) continue;
        int slot = kTBigs;
        if (c1 - c0 > kTAlone) {
          if (lane == 0) slot = atomicAdd(&ts.n_big, 1);
          slot = __shfl_sync(kFull, slot, 0);
        }
        if (slot < kTBigs) {
          if (lane == 0) ts.big[slot] = b0 + i;
        } else {
          walk_alone<MODE>(a, ts, b0 + i, c0, c1 - c0);
        }
      }
    }
    __syncwarp();
    t = tn;
    b0 = n0;
    b1 = n1;
    r0 = nr0;
    r1 = nr1;
  }

  if (bad) flag(a.status, kStatusData);
  __syncthreads();
  const int nbig = min(ts.n_big, kTBigs);
  if (nbig > 0) {
    // by warps, teams or the CTA, as walk_queue; more than a warp each only where none is large
    int64_t c0 = 0, n = 0;
    if (tid < nbig) batch_range(a, ts.big[tid], &c0, &n);
    const bool large = __syncthreads_or(n > kQTeam);
    if (queued && nbig > kTWarps) {
      walk_list<MODE, 32>(a, ts, nbig);
    } else if (!large && nbig >= kTTeams) {
      walk_list<MODE, kTTeam>(a, ts, nbig);
    } else {
      walk_list<MODE, kTThreads>(a, ts, nbig);
    }
  }
  if (queued && (ts.queued[0] | ts.queued[1] | ts.queued[2])) walk_queue<MODE>(a, ts);
  if (kTen) {
    __syncthreads();
    ten_table_flush(tw, kHotMax, a.H, a.ten_pend, tid, kTThreads);
    if (a.ten_state) ten_fold_last(a.ten_pend, a.ten_state, a.ten_ticket, a.n_tenants, a.status, tid, kTThreads);
  }
}

}  // namespace lv
