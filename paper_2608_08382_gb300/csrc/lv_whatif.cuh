// What-if evaluation over (pending request x candidate batch) pairs (Section 1:
// "what-if" planning over alternative batch mixes, admission control).
//
// For candidate batch b with sums (S1, S2, S3, n) and pending request j with
// (p, c), the batch b + {j} has sums (S1 + p, S2 + c, S3 + p^2, n + 1) and its
// phase is prefill if either side is.  With s the segment of b + {j}, Eq. 1 and
// j's share regroup as
//     T  = [beta + a1 S1 + a2 S2 + a3 S3 + a4 (n+1)^2]  +  [a1 p + a2 c + a3 p^2]
//        =            U_b[s]                            +         V_j[s]
//     t_j = [fl(beta/(n+1)) + fl(a4 (n+1))]             +         V_j[s]
//        =            W_b[s]                            +         V_j[s]
// U, W and V are exact 128-bit fixed-point values, formed for all four segments
// once per candidate (U, W) and once per block of pairs and row (V), so every
// pair costs a segment select, two exact additions and two roundings.  In fp64
// mode (or outside the exact range) a pair is evaluated left to right in double
// like any other batch.
#pragma once

#include "lv_kernels.cuh"
#include "lv_step.cuh"
#include "lv_tile.cuh"

namespace lv {

struct CandP {
  i128 U[4];
  i128 W[4];
  int64_t s1, s2, s3, n;
  int32_t prefill;
  int32_t slow;  // 1: evaluate pairs of this candidate in fp64
};

// A pending request in a block of pairs.
struct PendP {
  uint4 V3[4];  // V's low three words
  i128 V[4];
  int32_t p, c, phase, slow;
  double Lu, Bu;  // admission: the request's tenant's running total and budget
  int64_t Bk;     // order_key of the budget, below every sum's where it is NaN
};

// Order of doubles as signed integers (not NaN; -0 below +0).
__device__ __forceinline__ int64_t order_key(double x) {
  const int64_t b = (int64_t)__double_as_longlong(x);
  return b ^ ((b >> 63) & INT64_MAX);
}
// The key of a bound that x <= bound is tested against: -0 taken as +0, NaN
// below everything.
__device__ __forceinline__ int64_t bound_key(double x) {
  return x != x ? INT64_MIN : order_key(__dadd_rn(x, 0.0));
}

// Admission inputs (null: plain what-if).  A pair (j, b) is admissible when
// L[u_j] + share_new[j][b] <= budget[u_j] (one fp64 addition) and
// T_new[j][b] <= slo (Section 1: what-if planning for admission control).
struct AdmitArgs {
  const int32_t *tenant;  // [n_pending]
  const double *L, *budget;  // [n_tenants]
  int32_t n_tenants;
  double slo;
  uint8_t *admit;  // [n_pending][n_cand]
};

// U_b[s] (half 0) or W_b[s] (half 1) of a candidate; *slow where the exact
// range does not hold it.
__device__ __forceinline__ i128 cand_const(const ModelP &mp, int s, int half, int64_t s1, int64_t s2, int64_t s3,
                                           int64_t n, bool *slow) {
  const int64_t n1 = n + 1;
  if (half) return batch_k(mp, s, n1, slow).kf;
  const SegFix &f = mp.fx[s];
  const uint64_t F4 = (uint64_t)n1 * (uint64_t)n1;
  if ((uint64_t)s1 > f.lim[0] || (uint64_t)s2 > f.lim[1] || (uint64_t)s3 > f.lim[2] || F4 > f.lim[3] ||
      n1 > 0x7fffffffll) {
    *slow = true;
    return mk128(0, 0);
  }
  i128 U = f.B;
  U = add128(U, mul128_u64(f.A1, (uint64_t)s1));
  U = add128(U, mul128_u64(f.A2, (uint64_t)s2));
  U = add128(U, mul128_u64(f.A3, (uint64_t)s3));
  return add128(U, mul128_u64(f.A4, F4));
}

// Candidates straight from their requests, one block each: block sums, then
// one thread per constant.  One launch in place of the tile bounds, the tile
// pass and k_wi_cand: a planning call's few hundred to few thousand candidates
// are bound by the chain of launches and of dependent loads (1,024
// candidates of 144 requests: 29 us for that chain).  With more than
// kWiDirectPerSm candidates per SM the tile pass, which packs batches, takes
// over (whole calls by blocks and by tiles: 1,024 candidates 27 and 35 us, 10,000
// 41.5 and 43.5, 40,000 83 and 56).
// A candidate is one block's chain of loads, so a few large ones (at most two per
// SM, of more than kWiWide requests each on average) get blocks of 512 threads
// with four 16-byte loads of every array in flight each: 24 candidates of 1e6
// requests 255 us, 1,310 with 128 threads and four 4-byte loads; one of 5e6 1.0
// ms, 2.3.  The others get 128 threads with two such loads, few enough registers
// for ten blocks per SM (5,000 of 3,000: 47 us, 111 with 512 threads).
constexpr int kWiDirectPerSm = 64, kWiWide = 4096;
template <int kThreads, int kQuads>
__global__ void __launch_bounds__(kThreads, kThreads == 128 ? 10 : 1)
    k_wi_cand_direct(ModelP mp, const int32_t *__restrict__ p,
                     const int32_t *__restrict__ c, const int32_t *__restrict__ ph, const int64_t *__restrict__ off,
                     int64_t n_req, int64_t nc, CandP *__restrict__ out, int *status) {
  let_next();
  __shared__ Sums red[kThreads / 32];
  const int64_t b = blockIdx.x;
  const int tid = threadIdx.x;
  int bad = 0;
  const int64_t o0 = off[b], o1 = off[b + 1];
  const int64_t r0 = clampi(o0, 0, n_req), r1 = clampi(o1, r0, n_req);
  if (r0 != o0 || r1 != o1 || (b == 0 && o0 != 0) || (b == nc - 1 && o1 != n_req)) bad = 1;
  Sums acc{0, 0, 0, 0};
  for (int64_t q0 = (r0 & ~(int64_t)3) + 4 * tid; q0 < r1; q0 += 4 * kQuads * kThreads) {
    Quad v[kQuads];  // all loads in flight
#pragma unroll
    for (int h = 0; h < kQuads; ++h) {
      const int64_t q = q0 + 4 * kThreads * h, left = n_req - q;
      v[h].p = v[h].c = v[h].x = make_int4(0, 0, 0, 0);
      if (q < r1) v[h] = load_quad<true>(p + q, c + q, ph + q, 0, left < 4 ? (int)left : 4);
    }
#pragma unroll
    for (int h = 0; h < kQuads; ++h) {
      const int64_t q = q0 + 4 * kThreads * h;
      if (q >= r1) break;
      int32_t pv[4] = {v[h].p.x, v[h].p.y, v[h].p.z, v[h].p.w}, cv[4] = {v[h].c.x, v[h].c.y, v[h].c.z, v[h].c.w},
              fv[4] = {v[h].x.x, v[h].x.y, v[h].x.z, v[h].x.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (q + k < r0 || q + k >= r1) pv[k] = cv[k] = fv[k] = 0;
        check_req(pv[k], cv[k], fv[k], &bad);
        acc.s1 += pv[k];
        acc.s2 += cv[k];
        acc.s3 += (int64_t)pv[k] * pv[k];
        acc.ph |= fv[k];
      }
    }
  }
  acc = warp_sum(acc);
  if ((tid & 31) == 0) red[tid >> 5] = acc;
  if (bad) flag(status, kStatusData);
  __syncthreads();
  if (tid >= 32) return;
  acc = red[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) acc = add_sums(acc, red[w]);
  bool slow = !mp.fixed;
  if (tid < 8 && mp.fixed) {
    const i128 v = cand_const(mp, tid & 3, tid >> 2, acc.s1, acc.s2, acc.s3, r1 - r0, &slow);
    (tid < 4 ? out[b].U : out[b].W)[tid & 3] = v;
  }
  slow = __any_sync(kFull, slow);
  if (tid == 0) {
    out[b].s1 = acc.s1;
    out[b].s2 = acc.s2;
    out[b].s3 = acc.s3;
    out[b].n = r1 - r0;
    out[b].prefill = acc.ph > 0 ? 1 : 0;
    out[b].slow = slow ? 1 : 0;
  }
}

// The same from batch sums and segment codes (the tile pass).
__global__ void k_wi_cand(ModelP mp, const int64_t *__restrict__ bfeat, const uint8_t *__restrict__ bseg,
                          int64_t nc, CandP *__restrict__ out) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= nc) return;
  CandP cp;
  cp.s1 = bfeat[b];
  cp.s2 = bfeat[nc + b];
  cp.s3 = bfeat[2 * nc + b];
  cp.n = bfeat[3 * nc + b];
  cp.prefill = (bseg[b] >> 1) & 1;
  bool slow = !mp.fixed;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    cp.U[s] = mp.fixed ? cand_const(mp, s, 0, cp.s1, cp.s2, cp.s3, cp.n, &slow) : mk128(0, 0);
    cp.W[s] = mp.fixed ? cand_const(mp, s, 1, cp.s1, cp.s2, cp.s3, cp.n, &slow) : mk128(0, 0);
  }
  cp.slow = slow ? 1 : 0;
  out[b] = cp;
}

// V * 2^E rounded to double: the leading-word rounding for the common
// magnitude 2^64 <= V < 2^96, the general rounding otherwise.
__device__ __forceinline__ double round_fix(i128 V, int E) {
  const uint32_t v3 = (uint32_t)(V.hi >> 32), v2 = (uint32_t)V.hi;
  if (v3 == 0u && v2 != 0u)
    return round_top((uint32_t)V.lo, (uint32_t)(V.lo >> 32), v2, (uint32_t)(E + 32) << 20);
  return fix_to_double(V, E).d;
}

// x + V, both below 2^95 and x at least 2^64, rounded (ebase as round_top's).
__device__ __forceinline__ double sum_round(const uint32_t *x, const uint4 &V, uint32_t ebase) {
  uint32_t v0, v1, v2;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=r"(v0), "=r"(v1), "=r"(v2)
      : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(V.x), "r"(V.y), "r"(V.z));
  return round_top(v0, v1, v2, ebase);
}

// Left-to-right fp64 evaluation of one pair (fp64 mode, or outside the exact range).
__device__ __noinline__ void wi_pair_slow(const ModelP &mp, int s, int64_t s1, int64_t s2, int64_t s3, int64_t n1,
                                          int32_t p, int32_t c, double *T, double *share) {
  const BatchAgg g{s1, s2, s3, n1, 1};
  *T = eq1_fp64(mp.coef[s], g);
  bool dummy = false;
  const KEntry e = batch_k(mp, s, n1, &dummy);
  *share = share_fp64(mp.coef[s], e.q, e.a4n, p, c);
}

constexpr int kWiThreads = 128;  // threads per block
constexpr int kWiRows = 32;      // pending requests per block, at most

// Pair grid: block (bx, by) covers candidates [bx * C, + C), C = 2^lc, and
// pending rows [j_base + by * rows, + rows); thread t takes candidate t mod C
// and every (128 / C)-th row.  Consecutive threads write consecutive
// candidates of a row, so the row-major [pending][candidate] outputs are
// coalesced.  The host picks C and rows so that few candidates or few rows
// still fill the chip (500 x 24 pairs: 15 us with 128 columns and 32 rows, 5.7
// so).  The block's rows get their V here, one thread per row and segment; a
// candidate's U and W of the segment in use stay in registers (they change with
// the row only where the merged batch crosses the split or turns prefill), so a
// pair reads one V from shared memory.  Bound by the integer ALU pipe (75 % busy
// at 65 % issue: about 129 warp instructions per 32 pairs, most of them the two
// roundings' shifts and logic), ahead of the stores, 16-17 B a pair (4.2e6 pairs,
// 67 MB into L2: 21.5 us, 24.4 with U and W read per pair).
__global__ void __launch_bounds__(kWiThreads) k_wi_pairs(ModelP mp, const CandP *cand, int64_t nc,
                                                         const int32_t *__restrict__ p_new,
                                                         const int32_t *__restrict__ c_new,
                                                         const int32_t *__restrict__ ph_new, int64_t np,
                                                         int64_t j_base, int lc, int rows_per_block, AdmitArgs adm,
                                                         double *__restrict__ T_new, double *__restrict__ share_new,
                                                         int *status) {
  __shared__ PendP sp[kWiRows];
  __shared__ int sE[4];
  const int tid = threadIdx.x;
  const int64_t j0 = j_base + blockIdx.y * (int64_t)rows_per_block;
  const int rows = (int)(np - j0 < rows_per_block ? np - j0 : rows_per_block);
  int rslow = 0;
  for (int i = tid; i < 4 * rows; i += kWiThreads) {
    const int r = i >> 2, s = i & 3;
    const int64_t j = j0 + r;
    int32_t p = p_new[j], c = c_new[j], ph = ph_new[j];
    int bad = 0;
    check_req(p, c, ph, &bad);
    const int slow = (!mp.fixed || p > kPMaxFix) ? 1 : 0;
    rslow |= slow;
    i128 V = mk128(0, 0);
    if (!slow) {
      const SegFix &f = mp.fx[s];
      V = mul128_u32(add128(f.A1, mul128_u32(f.A3, (uint32_t)p)), (uint32_t)p);
      V = add128(V, a2_times(f, (uint32_t)c));
    }
    sp[r].V[s] = V;
    sp[r].V3[s] = make_uint4((uint32_t)V.lo, (uint32_t)(V.lo >> 32), (uint32_t)V.hi, 0u);
    rslow |= V.hi >= (1ull << 31) ? 1 : 0;
    if (s == 0) {
      sp[r].p = p;
      sp[r].c = c;
      sp[r].phase = ph;
      sp[r].slow = slow;
      if (adm.admit) {
        // a tenant id out of range, and a total that is a NaN of either sign, make
        // every pair of the request inadmissible: a NaN budget compares false, and
        // with the total at infinity no sum's key is as low as its bound's
        const int32_t u = adm.tenant[j];
        const bool in = u >= 0 && u < adm.n_tenants;
        if (!in) bad = 1;
        const double Lu = in ? adm.L[u] : 0.0;
        const bool ok = in && Lu == Lu;
        sp[r].Lu = ok ? Lu : __longlong_as_double(0x7ff0000000000000ll);
        sp[r].Bu = ok ? adm.budget[u] : __longlong_as_double(0x7ff8000000000000ll);
        sp[r].Bk = bound_key(sp[r].Bu);
      }
      if (bad) flag(status, kStatusData);
    }
  }
  if (tid < 4) sE[tid] = mp.fx[tid].E;
  rslow = __syncthreads_or(rslow);
  wait_previous();  // the candidates' kernel: the rows above do not need it
  const int64_t b = ((int64_t)blockIdx.x << lc) + (tid & ((1 << lc) - 1));
  if (b >= nc) return;
  const CandP *cb = cand + b;
  const int64_t s1 = cb->s1, sp0 = mp.split[0], sp1 = mp.split[1];
  const int prefill = cb->prefill, step = kWiThreads >> lc;
  int64_t o = (j0 + (tid >> lc)) * nc + b;
  const int64_t ostep = step * nc;
  if (!cb->slow && !rslow) {
    // every V of the block below 2^95 and p at most 2^24: with U and W in
    // [2^64, 2^95), three words hold the sums and one rounding form does
    // s1 + p >= split as p >= split - s1; a negative split, met by every batch,
    // counts as 0, so that the difference cannot wrap
    const int32_t thr0 = (int32_t)clampi(max(sp0, (int64_t)0) - s1, INT32_MIN, INT32_MAX),
                  thr1 = (int32_t)clampi(max(sp1, (int64_t)0) - s1, INT32_MIN, INT32_MAX);
    const int64_t slo_key = bound_key(adm.slo);
    double *Tp = T_new ? T_new + o : nullptr, *Sp = share_new ? share_new + o : nullptr;
    uint8_t *Ap = adm.admit ? adm.admit + o : nullptr;
    int cur = -1;
    uint32_t u[3] = {0u, 0u, 0u}, w[3] = {0u, 0u, 0u}, eb = 0u;
    bool narrow = false;
#pragma unroll 4
    for (int r = tid >> lc; r < rows; r += step) {
      const int phase = prefill | sp[r].phase;
      const int s = phase * 2 + (sp[r].p >= (phase ? thr1 : thr0) ? 1 : 0);
      if (s != cur) {
        cur = s;
        const i128 U = cb->U[s], W = cb->W[s];
        u[0] = (uint32_t)U.lo, u[1] = (uint32_t)(U.lo >> 32), u[2] = (uint32_t)U.hi;
        w[0] = (uint32_t)W.lo, w[1] = (uint32_t)(W.lo >> 32), w[2] = (uint32_t)W.hi;
        eb = (uint32_t)(sE[s] + 32) << 20;
        narrow = U.hi - 1ull < (1ull << 31) - 1ull && W.hi - 1ull < (1ull << 31) - 1ull;
      }
      const uint4 V = sp[r].V3[s];
      double T = sum_round(u, V, eb), sh = sum_round(w, V, eb);
      if (!narrow) {
        T = round_fix(add128(cb->U[s], sp[r].V[s]), sE[s]);
        sh = round_fix(add128(cb->W[s], sp[r].V[s]), sE[s]);
      }
      if (Tp) {
        __stcs(Tp, T);
        Tp += ostep;
      }
      if (Sp) {
        __stcs(Sp, sh);
        Sp += ostep;
      }
      // comparisons as integers: with two fp64 ones per pair as well as the
      // addition, the fp64 pipe took longer than all the rest (4.2e6 pairs: 52
      // us a call, 34 so).  No sum is a NaN: totals are not (above), shares are finite.
      if (Ap) {
        *Ap = (order_key(__dadd_rn(sp[r].Lu, sh)) <= sp[r].Bk && order_key(T) <= slo_key) ? 1 : 0;
        Ap += ostep;
      }
    }
    return;
  }
  const int64_t s2 = cb->s2, s3 = cb->s3, n1 = cb->n + 1;
  for (int r = tid >> lc; r < rows; r += step, o += ostep) {
    const int32_t p = sp[r].p, c = sp[r].c;
    const int phase = (prefill | sp[r].phase) ? 1 : 0;
    const int s = phase * 2 + ((s1 + p >= (phase ? sp1 : sp0)) ? 1 : 0);
    double T, sh;
    if (cb->slow | sp[r].slow) {
      wi_pair_slow(mp, s, s1 + p, s2 + c, s3 + (int64_t)p * p, n1, p, c, &T, &sh);
    } else {
      const i128 V = sp[r].V[s];
      T = round_fix(add128(cb->U[s], V), sE[s]);
      sh = round_fix(add128(cb->W[s], V), sE[s]);
    }
    if (T_new) __stcs(T_new + o, T);
    if (share_new) __stcs(share_new + o, sh);
    if (adm.admit) adm.admit[o] = (__dadd_rn(sp[r].Lu, sh) <= sp[r].Bu && T <= adm.slo) ? 1 : 0;
  }
}

}  // namespace lv
