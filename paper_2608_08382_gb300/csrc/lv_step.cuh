// Share arithmetic common to the request kernels, and the one-cluster kernel of
// a serving step (sm_103a).
#pragma once

#include <cooperative_groups.h>

#include "lv_kernels.cuh"

namespace lv {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ Sums add_sums(Sums a, const Sums &b) {
  a.s1 += b.s1;
  a.s2 += b.s2;
  a.s3 += b.s3;
  a.ph += b.ph;
  return a;
}

__device__ __forceinline__ Sums warp_sum(Sums v) {
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    v.s1 += __shfl_xor_sync(kFull, v.s1, d);
    v.s2 += __shfl_xor_sync(kFull, v.s2, d);
    v.s3 += __shfl_xor_sync(kFull, v.s3, d);
    v.ph += __shfl_xor_sync(kFull, v.ph, d);
  }
  return v;
}

// ---------------------------------------------------------------- decode fast path
//
// A decode request (p = 1) of a batch with constant K has the exact share
// V = K13 + A2 c with K13 = K + A1 + A3.  When A2 < 2^64 (the segment's
// a2_narrow) this is one 64x32-bit product and a 128-bit add; the result is
// rounded to double with 32-bit funnel shifts.  A prefill takes the same steps
// with K + p (A1 + A3 p) in place of K13 (prefill_const) where that is exact;
// the general path is exact for every case.

// v = k + (a1:a0) * c, four 32-bit words, exact (the sum stays below 2^128):
// carry-propagating multiply-adds, low word first.
__device__ __forceinline__ void mad_k13(uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3, uint32_t a0, uint32_t a1,
                                        uint32_t c, uint32_t &v0, uint32_t &v1, uint32_t &v2, uint32_t &v3) {
  asm("mad.lo.cc.u32 %0, %4, %6, %7;\n\t"
      "madc.hi.cc.u32 %1, %4, %6, %8;\n\t"
      "addc.cc.u32 %2, %9, 0;\n\t"
      "addc.u32 %3, %10, 0;\n\t"
      "mad.lo.cc.u32 %1, %5, %6, %1;\n\t"
      "madc.hi.cc.u32 %2, %5, %6, %2;\n\t"
      "addc.u32 %3, %3, 0;"
      : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3)
      : "r"(a0), "r"(a1), "r"(c), "r"(k0), "r"(k1), "r"(k2), "r"(k3));
}

// Constant part of a prefill request's share, kf + p (A1 + A3 p), for a
// segment with p_narrow and p <= 2^24: A1 + A3 p < 2^96 and its product with p
// stays below 2^120, so the 128-bit sum is exact whenever the share itself is
// below 2^128 (which the caller's V < 2^96 test then confirms).
__device__ __forceinline__ void prefill_const(const SegS &sg, i128 kf, uint32_t p, uint32_t &b0, uint32_t &b1,
                                              uint32_t &b2, uint32_t &b3) {
  const i128 r = add128(sg.A1, mul_u64_u32(sg.A3.lo, p));
  const i128 b = add128(kf, mul128_u32(r, p));
  b0 = (uint32_t)b.lo;
  b1 = (uint32_t)(b.lo >> 32);
  b2 = (uint32_t)b.hi;
  b3 = (uint32_t)(b.hi >> 32);
}

// Tenant contribution of a share m * 2^ex2 (m <= 2^53) when q = m 2^(ex2+72)
// has at most three 32-bit words and the tenant id is valid; false otherwise
// (nothing is added then).  Hot tenants: exact multi-word add in shared memory;
// cold tenants: 32-bit limbs into the global 64-bit pending counters.
__device__ __forceinline__ bool tenant_fast(const TileArgs &a, uint32_t *tt, int32_t u, uint64_t m, int ex2) {
  const int sh = ex2 - kTenLsb;
  if ((unsigned)sh <= 10u && (unsigned)u < (unsigned)a.H) {
    // the common case: q = m 2^sh <= 2^63, two words
    const uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
    uint32_t *w = ten_word0(tt, a.H, u);
    const int P = ten_plane(a.H);
    const uint32_t lo = ml << sh, hi = __funnelshift_l(ml, mh, sh);
    const uint32_t o0 = atomicAdd(w, lo);
    const uint32_t a1 = hi + ((o0 + lo < o0) ? 1u : 0u);  // hi <= 2^31: no wrap
    const uint32_t o1 = atomicAdd(w + P, a1);
    if (o1 + a1 < o1) {
      if (atomicAdd(w + 2 * P, 1u) == 0xffffffffu) atomicAdd(w + 3 * P, 1u);
    }
    return true;
  }
  if ((unsigned)sh > 42u || (unsigned)u >= (unsigned)a.n_tenants) return false;
  const uint32_t ml = (uint32_t)m, mh = (uint32_t)(m >> 32);
  const bool lowp = sh < 32;
  const int t = lowp ? sh : sh - 32;
  const uint32_t x0 = ml << t, x1 = __funnelshift_l(ml, mh, t), x2 = t ? mh >> (32 - t) : 0u;
  const uint32_t q0 = lowp ? x0 : 0u, q1 = lowp ? x1 : x0, q2 = lowp ? x2 : x1;
  if (u < a.H) {
    uint32_t *w = ten_word0(tt, a.H, u);
    const int P = ten_plane(a.H);
    const uint32_t o0 = atomicAdd(w, q0);
    const uint32_t a1 = q1 + ((o0 + q0 < o0) ? 1u : 0u);
    const uint32_t o1 = atomicAdd(w + P, a1);
    const uint32_t a2 = q2 + (((o1 + a1 < o1) || a1 < q1) ? 1u : 0u);  // q2 < 2^22: no wrap
    if (a2) {
      if (atomicAdd(w + 2 * P, a2) + a2 < a2) atomicAdd(w + 3 * P, 1u);
    }
  } else {
    unsigned long long *pw = a.ten_pend + 4 * (int64_t)u;
    atomicAdd(pw, (unsigned long long)q0);
    atomicAdd(pw + 1, (unsigned long long)q1);
    if (q2) atomicAdd(pw + 2, (unsigned long long)q2);
  }
  return true;
}

// One request's share, its store and its tenant contribution.
template <int MODE>
__device__ __forceinline__ void attribute_one(const TileArgs &a, uint32_t *tt, const SegS &sg, int s, bool slow,
                                              i128 kf, int64_t n, int64_t i, int32_t p, int32_t c, int32_t u,
                                              int *bad) {
  Rounded r;
  if ((MODE & M_FIX) && !slow && p <= kPMaxFix)
    r = share_fix(sg, kf, (uint32_t)p, (uint32_t)c);
  else
    r = share_slow(a.mp, s, (MODE & M_FIX) != 0, kf, p, c, n);
  if (a.share) __stcs(a.share + i, r.d);
  if (MODE & M_TEN) tenant_add(a, tt, u, r, bad);
}

// Per-request constant of a batch: fixed-point K, or {fl(beta/n), fl(a4 n)} in
// fp64 mode.
template <int MODE>
__device__ __forceinline__ i128 batch_const_w(const TileArgs &a, int s, int64_t n, bool *slow) {
  if (MODE & M_FIX) return batch_k(a.mp, s, n, slow).kf;
  bool dummy = false;
  const KEntry e = batch_k(a.mp, s, n, &dummy);
  return mk128((uint64_t)__double_as_longlong(e.q), (uint64_t)__double_as_longlong(e.a4n));
}

// Per-segment share parameters of a CTA.
template <int MODE>
__device__ __forceinline__ void init_segs(const TileArgs &a, SegS *seg) {
  if (threadIdx.x < 4) {
    const SegFix &f = a.mp.fx[threadIdx.x];
    SegS g;
    g.A1 = f.A1;
    g.A3 = f.A3;
    g.A13 = f.A13;
    g.A2 = f.A2;
    g.E = f.E;
    g.a2_narrow = f.a2_narrow;
    g.p_narrow = ((uint64_t)f.A1.hi < (1ull << 31) && f.A3.hi == 0) ? 1 : 0;
    g.t32 = seg_t32(f);
    seg[threadIdx.x] = g;
  }
}

// ---------------------------------------------------------------- small inputs

// A serving scheduler attributes one step's batches (a few thousand requests)
// at a time, where launch latency, not bandwidth, bounds the call.  For such
// inputs lv_attribute and lv_attribute_step run this kernel instead of the
// bounds, tile, fold and totals kernels: one cluster of kStepCtas
// CTAs with one request per thread (CTA r takes the r-th contiguous share of
// the requests) and one more warp per CTA for the batch constant.  The CTAs
// exchange partial results by asynchronous stores into one another's shared
// memory, each completing bytes on the receiver's transaction barrier, so no
// step waits at a cluster-wide barrier.
//   1. Thread 0 sets up the two receive barriers (the batch sums, the tenant
//      slice), and the cluster's threads arrive once on the cluster barrier,
//      which they wait for only before their first remote store.  Every global
//      read is issued at once: the thread's request, the offsets (warp 0
//      clamps them into non-decreasing batch bounds with a max-scan), and the
//      state of the tenants this CTA folds; each CTA zeroes its tenant table.
//      The constant warp meanwhile forms the per-request constant of a batch
//      of n_req requests for all four segments (the single-batch step's).
//   2. Per-batch sums of the CTA's requests: a warp whose requests share one
//      batch (the common case) keeps its warp sums (hardware reductions when
//      they fit 31 bits), a warp that spans a batch bound adds lane by lane
//      with shared atomics.  The CTA's sums go to every CTA of the cluster.
//   3. One thread per batch adds the CTAs' partial sums as they arrive and
//      picks the segment and the constant.
//   4. Every thread attributes its request and adds its share into the CTA's
//      exact tenant table; the constant warp of CTA 0 writes T.
//   5. Tenant u's table entry goes to the CTA that owns u's slice; there one
//      thread per tenant adds the cluster's entries exactly, and the tenant's
//      state (zero on a reset) is added, stored and, when asked, converted to
//      the correctly rounded total.
// A CTA leaves only after every byte addressed to it has arrived.  Each wait
// on a receive barrier is bounded (a few seconds); one that runs out records
// a timeout in the status word.  Tenant ids from H up still go to the pending
// limbs, which the caller folds.
constexpr int kStepCtas = 8;
constexpr int kStepThreads = 512;                 // request threads
constexpr int kStepBlock = kStepThreads + 32;     // and the constant warp
constexpr int64_t kSmallMaxReq = (int64_t)kStepCtas * kStepThreads;
constexpr int64_t kSmallMaxBatch = 16;
constexpr int kStepSlice = (kHotMax + kStepCtas - 1) / kStepCtas;  // tenants a CTA folds, at most
static_assert(kSmallMaxBatch < 32, "warp 0 scans the offsets");
static_assert(kStepThreads >= kStepSlice, "one thread per tenant of a slice");
static_assert(kStepThreads >= kStepCtas * kSmallMaxBatch * 4, "one remote store per thread sends the sums");
static_assert(kStepThreads >= kHotMax, "one thread per tenant sends the table");

struct StepSmem {
  alignas(16) SegS seg[4];
  alignas(16) i128 kspec[4];                                // constant of a batch of n_req requests, per segment
  alignas(16) i128 bk[kSmallMaxBatch];                      // each batch's constant
  alignas(16) unsigned long long sum[kSmallMaxBatch][4];     // requests of warps that span a batch bound
  alignas(16) unsigned long long wsum[kStepThreads / 32][4];  // each warp's sums (warps within one batch)
  alignas(16) unsigned long long rsum[kStepCtas][kSmallMaxBatch][4];  // every CTA's, as received
  alignas(16) int64_t cb[kSmallMaxBatch + 1];               // clamped batch bounds
  alignas(8) unsigned long long mbar[2];                    // receive barriers: sums, tenant slice
  alignas(16) BatchAgg agg[kSmallMaxBatch];                 // each batch's totals
  int kspec_slow[4];
  int bs[kSmallMaxBatch], bslow[kSmallMaxBatch];
  int wb[kStepThreads / 32];                                // batch of warp wsum[w], or -1
  int pad[3];
};
static_assert(sizeof(StepSmem) % 16 == 0, "the tenant table follows StepSmem");

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// The address of shared-memory address `a` in the CTA of cluster rank `rank`.
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, int rank) {
  uint32_t d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
  return d;
}

// A receive barrier of one phase: one arrival (here) and `bytes` to come.
__device__ __forceinline__ void rx_init(uint32_t mb, uint32_t bytes) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mb) : "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes) : "memory");
}

// 8 or 16 bytes into a peer's shared memory, completing as many bytes on the
// peer's barrier `rmb`.
__device__ __forceinline__ void rx_put64(uint32_t raddr, uint64_t v, uint32_t rmb) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(raddr), "l"(v),
               "r"(rmb)
               : "memory");
}
__device__ __forceinline__ void rx_put128(uint32_t raddr, i128 v, uint32_t rmb) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                   raddr),
               "r"((uint32_t)v.lo), "r"((uint32_t)(v.lo >> 32)), "r"((uint32_t)v.hi), "r"((uint32_t)(v.hi >> 32)),
               "r"(rmb)
               : "memory");
}

// Waits for the receive barrier's first phase (bounded: false when it ran
// out, after a few seconds); what arrived is then visible to this thread.
// Each try suspends the thread until the phase completes or about a
// microsecond has passed.
__device__ __forceinline__ bool rx_wait(uint32_t mb) {
  for (int k = 0; k < (1 << 22); ++k) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0, %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(mb), "n"(1000)
        : "memory");
    if (done) return true;
  }
  return false;
}

// This warp's contribution to the per-batch sums: when every active lane is
// in one batch (the common case), the warp's sums go to wsum[warp] (four
// hardware reductions when every sum fits 31 bits); otherwise each lane adds
// its fields to sum[its batch] with shared atomics.
__device__ __forceinline__ void step_sums(StepSmem &ss, bool at, int b, int32_t p, int32_t c, int32_t ph, int lane,
                                          int wid) {
  const unsigned am = __ballot_sync(kFull, at);
  const int b0 = am ? __shfl_sync(kFull, b, __ffs(am) - 1) : -1;
  if (__all_sync(kFull, !at || b == b0)) {
    unsigned long long w[4];
    if (__all_sync(kFull, (uint32_t)p < (1u << 13) && (uint32_t)c < (1u << 26))) {
      w[0] = __reduce_add_sync(kFull, at ? (uint32_t)p : 0u);
      w[1] = __reduce_add_sync(kFull, at ? (uint32_t)c : 0u);
      w[2] = __reduce_add_sync(kFull, at ? (uint32_t)(p * p) : 0u);
      w[3] = __reduce_add_sync(kFull, at ? (uint32_t)ph : 0u);
    } else {
      Sums v{at ? p : 0, at ? c : 0, at ? (int64_t)p * p : 0, at ? ph : 0};
      v = warp_sum(v);
      w[0] = (unsigned long long)v.s1;
      w[1] = (unsigned long long)v.s2;
      w[2] = (unsigned long long)v.s3;
      w[3] = (unsigned long long)v.ph;
    }
    if (lane == 0) {
      ss.wb[wid] = b0;
#pragma unroll
      for (int k = 0; k < 4; ++k) ss.wsum[wid][k] = w[k];
    }
  } else {
    if (lane == 0) ss.wb[wid] = -1;
    if (at) {
      atomicAdd(&ss.sum[b][0], (unsigned long long)p);
      atomicAdd(&ss.sum[b][1], (unsigned long long)c);
      atomicAdd(&ss.sum[b][2], (unsigned long long)((int64_t)p * p));
      atomicAdd(&ss.sum[b][3], (unsigned long long)ph);
    }
  }
}

// Barrier of the request threads alone (the constant warp does not wait).
__device__ __forceinline__ void sync_requests() { asm volatile("bar.sync 1, %0;" ::"n"(kStepThreads) : "memory"); }

// state: the tenant accumulator's exact state (with M_TEN); L: the tenants'
// totals after this step, or null (then tenant ids may exceed H); reset: the
// state is taken as zero.
template <int MODE>
__global__ void __cluster_dims__(kStepCtas, 1, 1) __launch_bounds__(kStepBlock)
    k_step(const TileArgs a, i128 *state, double *L, int reset) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  StepSmem &ss = *reinterpret_cast<StepSmem *>(smem_raw);
  uint32_t *tt = reinterpret_cast<uint32_t *>(smem_raw + sizeof(StepSmem));
  constexpr bool kTen = (MODE & M_TEN) != 0;
  const int TS = kTen ? (a.H + kStepCtas - 1) / kStepCtas : 0;  // tenants per slice
  i128 *rt = reinterpret_cast<i128 *>(smem_raw + sizeof(StepSmem) + (kTen ? ten_bytes(a.H) : 0));  // [src][TS]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int r = (int)cooperative_groups::this_cluster().block_rank();
  const int64_t nr = a.n_req, nb = a.n_batch;
  const bool req = tid < kStepThreads;
  const uint32_t mb0 = smem_u32(&ss.mbar[0]), mb1 = smem_u32(&ss.mbar[1]);
  int bad = 0;

  // 1. receive barriers, reads, the single-batch constant
  const int own = kTen ? max(0, min(TS, a.H - r * TS)) : 0;  // tenants of this CTA's slice
  if (tid == 0) {
    rx_init(mb0, (uint32_t)(kStepCtas * 32 * nb));
    rx_init(mb1, (uint32_t)(kStepCtas * 16 * own));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
  const int64_t chunk = (nr + kStepCtas - 1) / kStepCtas;
  const int64_t i = r * chunk + tid;
  const bool in = req && tid < chunk && i < nr;
  int32_t p = 0, c = 0, ph = 0, u = 0;
  if (in) {
    p = a.p[i];
    c = a.c[i];
    ph = a.ph[i];
    if (kTen) u = a.ten[i];
  }
  int64_t ob = 0;
  if (wid == 0 && lane <= nb) ob = a.off[lane];
  // the fold: thread j takes tenant r * TS + j of this CTA's slice
  const int v = r * TS + tid;
  const bool fv = tid < own;
  i128 st0 = mk128(0, 0);
  if (fv && !reset) st0 = state[v];
  if (!req) {
    if (lane < 4) {
      bool slow = false;
      ss.kspec[lane] = nr > 0 ? batch_const_w<MODE>(a, lane, nr, &slow) : mk128(0, 0);
      ss.kspec_slow[lane] = slow ? 1 : 0;
    }
  } else {
    if (kTen)
      for (int k = tid; k < 4 * ten_plane(a.H); k += kStepThreads) tt[k] = 0;
    if (tid < 4 * kSmallMaxBatch) (&ss.sum[0][0])[tid] = 0ull;
    init_segs<MODE>(a, ss.seg);
    if (in) check_req(p, c, ph, &bad);
    if (wid == 0) {
      // bound k = min(n_req, max(0, off[0..k])): batch b takes requests
      // [cb[b], cb[b + 1]); valid offsets are their own bounds
      int64_t m = lane <= nb ? max(ob, (int64_t)0) : 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int64_t o = __shfl_up_sync(kFull, m, d);
        if (lane >= d) m = max(m, o);
      }
      m = min(m, nr);
      if (lane <= nb) {
        ss.cb[lane] = m;
        if (r == 0 && (m != ob || (lane == 0 && ob != 0) || (lane == nb && ob != nr))) bad = 1;
      }
    }
    sync_requests();

    // 2. per-batch sums, sent to every CTA of the cluster
    int b = 0;
    for (int k = 1; k < nb; ++k) b += ss.cb[k] <= i ? 1 : 0;
    const bool at = in && i >= ss.cb[0] && i < ss.cb[nb];
    step_sums(ss, at, b, p, c, ph, lane, wid);
    sync_requests();
    asm volatile("barrier.cluster.wait;" ::: "memory");  // the peers' receive barriers are set up
    if (tid < kStepCtas * 4 * nb) {
      // word k of the CTA's batch sums (batch k / 4), to CTA dst
      const int dst = tid / (4 * (int)nb), k = tid % (4 * (int)nb), kb = k >> 2, kw = k & 3;
      unsigned long long x = ss.sum[kb][kw];
#pragma unroll
      for (int j = 0; j < kStepThreads / 32; ++j) x += ss.wb[j] == kb ? ss.wsum[j][kw] : 0ull;
      rx_put64(peer_addr(smem_u32(&ss.rsum[r][kb][kw]), dst), x, peer_addr(mb0, dst));
    }
    // each request thread keeps its batch index in p's place until step 4
    ph = at ? b : -1;
  }
  __syncthreads();

  // 3. the batches' totals, segment, T and constant
  if (tid < nb) {
    if (!rx_wait(mb0)) flag(a.status, kStatusTimeout);
    unsigned long long t[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int src = 0; src < kStepCtas; ++src)
#pragma unroll
      for (int w = 0; w < 4; ++w) t[w] += ss.rsum[src][tid][w];
    const int64_t n = ss.cb[tid + 1] - ss.cb[tid];
    const BatchAgg g{(int64_t)t[0], (int64_t)t[1], (int64_t)t[2], n, t[3] > 0};
    const int s = segment_of(a.mp, g);
    ss.agg[tid] = g;
    bool slow = false;
    i128 kf = mk128(0, 0);
    if (n == nr) {
      kf = ss.kspec[s];
      slow = ss.kspec_slow[s] != 0;
    } else if (n > 0) {
      kf = batch_const_w<MODE>(a, s, n, &slow);
    }
    ss.bs[tid] = s;
    ss.bk[tid] = kf;
    ss.bslow[tid] = slow ? 1 : 0;
  }
  __syncthreads();

  // 4. this thread's request; T from the constant warp of CTA 0
  if (!req) {
    if (r == 0 && lane < nb) emit_batch<MODE>(a, lane, ss.agg[lane], ss.bs[lane], a.mp.fx);
  } else if (ph >= 0) {
    const int b = ph;
    const int s = ss.bs[b];
    const bool slow = ss.bslow[b] != 0;
    const i128 kf = ss.bk[b];
    const SegS sg = ss.seg[s];
    bool done = false;
    if ((MODE & M_FIX) && !slow && sg.a2_narrow && (p == 1 || (sg.p_narrow && p <= kPMaxFix))) {
      // the exact steps of the warp-tile fast path, with K + A1 + A3 for a
      // decode request and K + p (A1 + A3 p) for a prefill (one instruction
      // stream for both: a branch to rarely run code fetches it cold)
      const i128 K13 = add128(kf, sg.A13);
      uint32_t b0, b1, b2, b3, v0, v1, v2, v3;
      prefill_const(sg, kf, sg.p_narrow ? (uint32_t)p : 1u, b0, b1, b2, b3);
      if (p == 1) {
        b0 = (uint32_t)K13.lo;
        b1 = (uint32_t)(K13.lo >> 32);
        b2 = (uint32_t)K13.hi;
        b3 = (uint32_t)(K13.hi >> 32);
      }
      mad_k13(b0, b1, b2, b3, (uint32_t)sg.A2.lo, (uint32_t)(sg.A2.lo >> 32), (uint32_t)c, v0, v1, v2, v3);
      if (v3 == 0u && v2 != 0u) {
        uint64_t m;
        int ex2;
        const double d = round96(v0, v1, v2, sg.E, m, ex2);
        if (!kTen || tenant_fast(a, tt, u, m, ex2)) {
          if (a.share) __stcs(a.share + i, d);
          done = true;
        }
      }
    }
    if (!done) attribute_one<MODE>(a, tt, sg, s, slow, kf, ss.cb[b + 1] - ss.cb[b], i, p, c, u, &bad);
  }
  if (bad) flag(a.status, kStatusData);

  // 5. each tenant's table entry to the CTA of its slice, then the fold there
  if constexpr (kTen) {
    __syncthreads();
    if (tid < a.H) {
      const int dst = tid / TS;
      rx_put128(peer_addr(smem_u32(&rt[r * TS + (tid - dst * TS)]), dst), hot_value(tt, a.H, tid),
                peer_addr(mb1, dst));
    }
    if (fv) {
      if (!rx_wait(mb1)) flag(a.status, kStatusTimeout);
      i128 tv = rt[tid];
#pragma unroll
      for (int src = 1; src < kStepCtas; ++src) tv = add128(tv, rt[src * TS + tid]);
      const i128 nw = add128(st0, tv);
      // overflow of the signed 128-bit total (|total| >= 2^127 * 2^-72 s)
      if (is_neg128(st0) == is_neg128(tv) && is_neg128(nw) != is_neg128(st0)) flag(a.status, kStatusData);
      if (reset || (tv.lo | tv.hi)) state[v] = nw;
      if (L) L[v] = fix_to_double(nw, kTenLsb).d;
    }
  }
}

}  // namespace lv
