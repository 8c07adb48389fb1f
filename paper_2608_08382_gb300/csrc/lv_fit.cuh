// Least-squares fit of Eq. 1's coefficients (Section 2.1: "ordinary least
// squares on profiling data", one coefficient set per phase and regime).
//
// For every group g (segment phase*2 + regime) the design rows are the batch
// sums x = [1, S1, S2, S3, n^2] of the profiled batches of that group and the
// targets are their measured latencies y.  The normal equations need the Gram
// matrix X^T X and X^T y per group.  Both are accumulated EXACTLY:
//   - X^T X in 128-bit integers (features are integers below 2^48, so each
//     product is below 2^96);
//   - X^T y in fixed point with y rounded to a multiple of 2^-100 s (exact for any
//     latency whose lowest bit is at least 2^-100 s), in 256 bits: a lane's and a
//     warp's sums in 192, which hold a launch's share of the batches.
// The tile kernel writes each batch's sums and segment, and k_fit_gram adds the
// products with one lane per batch.  CTA partials are reduced exactly (integer
// adds) and each group's small system is solved in double-double (about
// 106-bit) arithmetic after power-of-two column scaling, with singular and
// under-determined groups reported.
#pragma once

#include "lv_kernels.cuh"

namespace lv {

// ---------------------------------------------------------------- products

// One row of blocks (blockIdx.y) per kind of entry: 0 the Gram matrix and the
// flag, 1 + k the latency vector k's X^T y and y'y.  For each group a warp
// collects the batches of that group in a queue and works them off 32 at a
// time, one batch per lane, its accumulators in registers (exact integers: the
// Gram's in 128 bits, X^T y modulo 2^192, y'y in 256).  Entry order
// in `partial`: 15 Gram pairs (a <= b, row order), 5 X^T y per y, one y'y per
// y, one flag (some batch has S1 != S3).
// Bound by latency at 16 warps per SM (128 registers): the products are chains of
// 32-bit multiply-adds through the carry, a quarter fewer instructions than
// 64-bit ones, issued in 57 % of the slots.  2e6 batches with two vectors take 111
// us; 150 with 64-bit products, 245 with, besides, one row of 32 segments looked at per turn and
// nothing loaded ahead.  With one entry per lane and all lanes on one batch,
// inside the kernel over the requests, the same sums took about 0.35 of 0.96 ms.
constexpr int kGramThreads = 256;
constexpr int kGramWarps = kGramThreads / 32;
constexpr int kGramMax = 16;  // entries of one row of blocks, at most
constexpr int kGramScan = 8;  // rows of 32 batches looked at together

// v += o for W 32-bit words (modulo 2^(32 W)).
template <int W>
__device__ __forceinline__ void add_words(uint32_t *v, const uint32_t *o) {
  static_assert(W == 3 || W == 4 || W == 6 || W == 8, "");
  if constexpr (W == 3)
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2])
        : "r"(o[0]), "r"(o[1]), "r"(o[2]));
  else if constexpr (W == 4)
    asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.cc.u32 %2, %2, %6;\n\taddc.u32 %3, %3, %7;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3])
        : "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]));
  else if constexpr (W == 6)
    asm("add.cc.u32 %0, %0, %6;\n\taddc.cc.u32 %1, %1, %7;\n\taddc.cc.u32 %2, %2, %8;\n\t"
        "addc.cc.u32 %3, %3, %9;\n\taddc.cc.u32 %4, %4, %10;\n\taddc.u32 %5, %5, %11;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5])
        : "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]));
  else
    asm("add.cc.u32 %0, %0, %8;\n\taddc.cc.u32 %1, %1, %9;\n\taddc.cc.u32 %2, %2, %10;\n\t"
        "addc.cc.u32 %3, %3, %11;\n\taddc.cc.u32 %4, %4, %12;\n\taddc.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\taddc.u32 %7, %7, %15;"
        : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
        : "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7]));
}

// Sum over the warp of a W-word integer (modulo 2^(32 W)), into dst (lane 0),
// sign-extended when `sign`.
template <int W>
__device__ __forceinline__ void warp_words(uint32_t *v, FitAcc *dst, bool sign, int lane) {
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    uint32_t o[W];
#pragma unroll
    for (int w = 0; w < W; ++w) o[w] = __shfl_xor_sync(0xffffffffu, v[w], d);
    add_words<W>(v, o);
  }
  if (lane == 0) {
    const uint32_t fill = sign && (int32_t)v[W - 1] < 0 ? ~0u : 0u;
#pragma unroll
    for (int w = 0; w < 4; ++w)
      dst->w[w] = (uint64_t)(2 * w < W ? v[2 * w < W ? 2 * w : 0] : fill) |
                  (uint64_t)(2 * w + 1 < W ? v[2 * w + 1 < W ? 2 * w + 1 : 0] : fill) << 32;
  }
}

// A feature below 2^48 in two words.
struct Feat48 {
  uint32_t l, h;
};

// a (4 words) += x y for x, y below 2^48.
__device__ __forceinline__ void mac48(uint32_t *a, Feat48 x, Feat48 y) {
  const uint64_t m = (uint64_t)x.l * y.h + (uint64_t)x.h * y.l;  // below 2^49
  asm("mad.lo.cc.u32 %0, %4, %5, %0;\n\t"
      "madc.hi.cc.u32 %1, %4, %5, %1;\n\t"
      "addc.cc.u32 %2, %2, 0;\n\t"
      "addc.u32 %3, %3, 0;\n\t"
      "add.cc.u32 %1, %1, %6;\n\t"
      "addc.cc.u32 %2, %2, %7;\n\t"
      "addc.u32 %3, %3, 0;"
      : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3])
      : "r"(x.l), "r"(y.l), "r"((uint32_t)m), "r"((uint32_t)(m >> 32) + x.h * y.h));
}

// a (6 words) += x Y modulo 2^192 for x below 2^48 and Y of four words, two's
// complement (neg: all ones where it is negative): Y as unsigned, less x 2^128.
__device__ __forceinline__ void mac48x128(uint32_t *a, Feat48 x, const uint32_t *Y, uint32_t neg) {
  asm("mad.lo.cc.u32 %0, %6, %8, %0;\n\t"
      "madc.hi.cc.u32 %1, %6, %8, %1;\n\t"
      "madc.lo.cc.u32 %2, %6, %10, %2;\n\t"
      "madc.hi.cc.u32 %3, %6, %10, %3;\n\t"
      "addc.cc.u32 %4, %4, 0;\n\t"
      "addc.u32 %5, %5, 0;\n\t"
      "mad.lo.cc.u32 %1, %6, %9, %1;\n\t"
      "madc.hi.cc.u32 %2, %6, %9, %2;\n\t"
      "madc.lo.cc.u32 %3, %6, %11, %3;\n\t"
      "madc.hi.cc.u32 %4, %6, %11, %4;\n\t"
      "addc.u32 %5, %5, 0;\n\t"
      "mad.lo.cc.u32 %1, %7, %8, %1;\n\t"
      "madc.hi.cc.u32 %2, %7, %8, %2;\n\t"
      "madc.lo.cc.u32 %3, %7, %10, %3;\n\t"
      "madc.hi.cc.u32 %4, %7, %10, %4;\n\t"
      "addc.u32 %5, %5, 0;\n\t"
      "mad.lo.cc.u32 %2, %7, %9, %2;\n\t"
      "madc.hi.cc.u32 %3, %7, %9, %3;\n\t"
      "madc.lo.cc.u32 %4, %7, %11, %4;\n\t"
      "madc.hi.u32 %5, %7, %11, %5;\n\t"
      "sub.cc.u32 %4, %4, %12;\n\t"
      "subc.u32 %5, %5, %13;"
      : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5])
      : "r"(x.l), "r"(x.h), "r"(Y[0]), "r"(Y[1]), "r"(Y[2]), "r"(Y[3]), "r"(x.l & neg), "r"(x.h & neg));
}

// A batch as loaded (n = 0: none).
struct GramRaw {
  int64_t s1, s2, s3, n;
  double y;
};

struct GramAcc {
  uint32_t lin[5][3];  // n, S1, S2, S3, n^2 (below 2^96: fewer than 2^48 batches)
  uint32_t sq[10][4];  // S1 S1, S1 S2, S1 S3, S1 n^2, S2 S2, ...
  bool flag;
};

struct FitYAcc {
  uint32_t xy[5][6];
  uint32_t yy[8];
};

__device__ __forceinline__ void gram_add(GramAcc &g, const Feat48 *x) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const uint32_t o[3] = {x[i].l, x[i].h, 0u};
    add_words<3>(g.lin[i], o);
  }
  int e = 0;
#pragma unroll
  for (int i = 1; i < 5; ++i)
#pragma unroll
    for (int j = i; j < 5; ++j, ++e) mac48(g.sq[e], x[i], x[j]);
  g.flag |= x[1].l != x[3].l || x[1].h != x[3].h;
}

__device__ __forceinline__ void fit_y_add(FitYAcc &g, const Feat48 *x, i128 Y) {
  uint32_t y[4] = {(uint32_t)Y.lo, (uint32_t)(Y.lo >> 32), (uint32_t)Y.hi, (uint32_t)(Y.hi >> 32)};
  const uint32_t neg = is_neg128(Y) ? ~0u : 0u;
  const uint32_t one[6] = {y[0], y[1], y[2], y[3], neg, neg};  // the column of ones (Y = 0 where there is no batch)
  add_words<6>(g.xy[0], one);
#pragma unroll
  for (int i = 1; i < 5; ++i) mac48x128(g.xy[i], x[i], y, neg);
  // y'y: Y^2 (below 2^250) shifted right by 64 bits
  if (neg) Y = neg128(Y);
  const uint64_t l = Y.lo, h = Y.hi;
  uint64_t w[4] = {__umul64hi(l, l), h * h, __umul64hi(h, h), 0ull};
  const uint64_t h0 = h * l, h1 = __umul64hi(h, l);
  acc_add256(w, h0 << 1, (h1 << 1) | (h0 >> 63), h1 >> 63, 0ull);
  const uint32_t o[8] = {(uint32_t)w[0], (uint32_t)(w[0] >> 32), (uint32_t)w[1], (uint32_t)(w[1] >> 32),
                         (uint32_t)w[2], (uint32_t)(w[2] >> 32), 0u, 0u};
  add_words<8>(g.yy, o);
}

// The batches of one launch.  Their sums and segments come from the tile kernel
// through a scratch of bounded size, so a fit of more than kFitRange batches is
// worked off in ranges of tiles that start in kFitRange batches each.  A range
// of 2^22 takes 138 MB and costs about 37 us (two launches, a search of the tiles,
// both kernels' ends): 8e6 batches of 1 to 64 requests 1,156 us, 1,117 with a
// scratch for all of them.
constexpr int64_t kFitRange = 1ll << 22;
// Rows of blocks, at least.  A product of a feature (below 2^48) and a latency
// (2^100 y, below 2^125) is below 2^173, so a warp's signed sum in 192 bits holds
// 2^18 of them; with this many rows a warp meets fewer than 2^17 + 2^10 batches
// of a range (the tiles that start in it reach less than 2^10 past it), rounded
// up to its turns of 2^8.
constexpr int kGramMinRows = 4;
static_assert(kFitRange / (kGramMinRows * kGramWarps) + (1 << 11) < (1 << 18), "X^T y of a warp fits 192 bits");
struct FitRange {
  const int64_t *feat;   // [4][stride] S1, S2, S3, n of batches lo and up
  const uint8_t *seg;    // [stride]
  int64_t stride, lo;
  int64_t n_batch;       // of the whole input (y's rows)
  const int64_t *range;  // first batch and the one past the last, from lo; null: all
};

struct GramSmem {
  int64_t queue[kGramWarps][32 * (kGramScan + 1)];
  FitAcc part[kGramWarps][kGramMax];
};

// kGram: the Gram matrix and the flag, else the latency vector k.
template <bool kGram>
__device__ __forceinline__ void fit_rows(GramSmem &sm, const FitRange &fr, const double *__restrict__ y, int n_y,
                                         int k, FitAcc *__restrict__ partial, int *status) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int NE = fit_entries(n_y);
  const int64_t stride = (int64_t)gridDim.x * kGramWarps * kGramScan * 32;
  int64_t *q = sm.queue[wid];
  int bad = 0;
  const int64_t *feat = fr.feat;
  const uint8_t *seg = fr.seg;
  const int64_t fs = fr.stride, first = fr.range ? fr.range[0] : 0, nb = fr.range ? fr.range[1] : fr.n_batch;
  const double *yk = y + (int64_t)k * fr.n_batch + fr.lo;
  int s[kGramScan];
  auto scan = [&](int64_t i0) {  // segments of kGramScan rows of 32 batches, their loads in flight together
#pragma unroll
    for (int r = 0; r < kGramScan; ++r) {
      const int64_t i = i0 + 32 * r + lane;
      s[r] = i < nb ? seg[i] : 255;
    }
  };
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    GramAcc ga{};
    FitYAcc ya{};
    GramRaw cur{0, 0, 0, 0, 0.0};
    auto add = [&]() {
      const uint64_t v[5] = {cur.n > 0 ? 1ull : 0ull, (uint64_t)cur.s1, (uint64_t)cur.s2, (uint64_t)cur.s3,
                             (uint64_t)cur.n * (uint64_t)cur.n};
      const bool ok = (v[1] | v[2] | v[3] | v[4]) < (uint64_t)kFitFeatMax && (uint64_t)cur.n < (1ull << 24);
      if (!ok) flag(status, kStatusOverflow);
      Feat48 x[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) x[c] = Feat48{ok ? (uint32_t)v[c] : 0u, ok ? (uint32_t)(v[c] >> 32) : 0u};
      if (kGram) {
        gram_add(ga, x);
      } else {
        bool ovf = false;
        const i128 Y = x[0].l ? double_to_fix(cur.y, kFitYLsb, &ovf) : mk128(0, 0);
        if (ovf) bad = 1;
        fit_y_add(ya, x, Y);
      }
    };
    int qn = 0;
    int64_t i0 = first + ((int64_t)blockIdx.x * kGramWarps + wid) * kGramScan * 32;
    scan(i0);
    while (i0 < nb || qn > 0) {
      const bool rest = i0 >= nb;  // no batches left: work off the queue
      if (!rest) {
#pragma unroll
        for (int r = 0; r < kGramScan; ++r) {
          const uint32_t m = __ballot_sync(0xffffffffu, s[r] == g);
          if (s[r] == g) q[qn + __popc(m & ((1u << lane) - 1u))] = i0 + 32 * r + lane;
          qn += __popc(m);
        }
        i0 += stride;
        scan(i0);  // for the next turn
        __syncwarp();
      }
#pragma unroll 1
      while (qn >= 32 || (rest && qn > 0)) {
        // the next 32 batches' values are loaded while the ones before them are added
        const int take = qn < 32 ? qn : 32;
        GramRaw nx{0, 0, 0, 0, 0.0};
        if (lane < take) {
          const int64_t b = q[qn - take + lane];
          nx.s1 = feat[b];
          nx.s2 = feat[fs + b];
          nx.s3 = feat[2 * fs + b];
          nx.n = feat[3 * fs + b];
          if (!kGram) nx.y = yk[b];
        }
        qn -= take;
        add();
        cur = nx;
      }
      __syncwarp();  // the queue's slots are written again
    }
    add();
    FitAcc *pw = sm.part[wid];
    int ne;
    if (kGram) {
      ne = 16;
#pragma unroll
      for (int i = 0; i < 5; ++i) warp_words<3>(ga.lin[i], pw + i, false, lane);
#pragma unroll
      for (int e = 0; e < 10; ++e) warp_words<4>(ga.sq[e], pw + 5 + e, false, lane);
      const bool any = __any_sync(0xffffffffu, ga.flag);
      if (lane == 0) pw[15] = FitAcc{{any ? 1ull : 0ull, 0ull, 0ull, 0ull}};
    } else {
      ne = 6;
#pragma unroll
      for (int i = 0; i < 5; ++i) warp_words<6>(ya.xy[i], pw + i, true, lane);
      warp_words<8>(ya.yy, pw + 5, false, lane);
    }
    __syncthreads();
    if ((int)threadIdx.x < ne) {
      const int e = threadIdx.x;
      const bool is_flag = kGram && e == 15;
      const int at = kGram ? (is_flag ? NE - 1 : e) : e < 5 ? 15 + 5 * k + e : 15 + 5 * n_y + k;
      FitAcc *out = partial + (int64_t)blockIdx.x * (4 * NE) + g * NE + at;
      FitAcc s{{0ull, 0ull, 0ull, 0ull}};
      if (fr.lo > 0) {  // added to what the ranges before gave
#pragma unroll
        for (int w = 0; w < 4; ++w) s.w[w] = __ldcg(reinterpret_cast<unsigned long long *>(out->w) + w);
      }
      for (int w = 0; w < kGramWarps; ++w) {
        const FitAcc &v = sm.part[w][e];
        if (is_flag)
          s.w[0] |= v.w[0];
        else
          acc_add256(s.w, v.w[0], v.w[1], v.w[2], v.w[3]);
      }
      *out = s;
    }
    __syncthreads();
  }
  if (bad) flag(status, kStatusData);
}

__global__ void __launch_bounds__(kGramThreads, 2)
    k_fit_gram(const FitRange fr, const double *__restrict__ y, int n_y, FitAcc *__restrict__ partial, int *status) {
  __shared__ GramSmem sm;
  let_next();
  wait_previous();
  if (blockIdx.y == 0)
    fit_rows<true>(sm, fr, y, n_y, 0, partial, status);
  else
    fit_rows<false>(sm, fr, y, n_y, (int)blockIdx.y - 1, partial, status);
}

// ---------------------------------------------------------------- reduction across CTAs

// totals[ge] = sum over CTAs of partial[cta][ge]: one block per entry, threads
// striding over the CTAs, then a tree in shared memory.  Integer addition is
// associative, so the exact result does not depend on the order; the flag
// entries are ORed.
constexpr int kFitRedThreads = 256;
__global__ void __launch_bounds__(kFitRedThreads) k_fit_reduce(const FitAcc *partial, int n_cta, int n_ent,
                                                               FitAcc *__restrict__ totals) {
  let_next();
  wait_previous();
  __shared__ FitAcc red[kFitRedThreads];
  const int ge = blockIdx.x;
  const bool is_flag = ge % (n_ent / 4) == n_ent / 4 - 1;
  FitAcc t;
  t.w[0] = t.w[1] = t.w[2] = t.w[3] = 0;
  for (int c = threadIdx.x; c < n_cta; c += kFitRedThreads) {
    const FitAcc p = partial[(int64_t)c * n_ent + ge];
    if (is_flag)
      t.w[0] |= p.w[0];
    else
      acc_add256(t.w, p.w[0], p.w[1], p.w[2], p.w[3]);
  }
  red[threadIdx.x] = t;
  __syncthreads();
  for (int h = kFitRedThreads / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      const FitAcc o = red[threadIdx.x + h];
      if (is_flag)
        red[threadIdx.x].w[0] |= o.w[0];
      else
        acc_add256(red[threadIdx.x].w, o.w[0], o.w[1], o.w[2], o.w[3]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) totals[ge] = red[0];
}

// ---------------------------------------------------------------- double-double arithmetic
// Error-free transformations (Knuth's two-sum, Dekker's product via FMA) and the
// usual double-double operations built on them.

struct dd {
  double hi, lo;
};

__device__ __forceinline__ dd two_sum(double a, double b) {
  const double s = __dadd_rn(a, b);
  const double bb = __dsub_rn(s, a);
  const double e = __dadd_rn(__dsub_rn(a, __dsub_rn(s, bb)), __dsub_rn(b, bb));
  return dd{s, e};
}

__device__ __forceinline__ dd quick_two_sum(double a, double b) {
  const double s = __dadd_rn(a, b);
  return dd{s, __dsub_rn(b, __dsub_rn(s, a))};
}

__device__ __forceinline__ dd dd_add(dd x, dd y) {
  dd s = two_sum(x.hi, y.hi);
  const dd t = two_sum(x.lo, y.lo);
  s.lo = __dadd_rn(s.lo, t.hi);
  s = quick_two_sum(s.hi, s.lo);
  s.lo = __dadd_rn(s.lo, t.lo);
  return quick_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ dd dd_neg(dd x) { return dd{-x.hi, -x.lo}; }

__device__ __forceinline__ dd dd_mul(dd x, dd y) {
  const double p = __dmul_rn(x.hi, y.hi);
  double e = __fma_rn(x.hi, y.hi, -p);
  e = __fma_rn(x.hi, y.lo, e);
  e = __fma_rn(x.lo, y.hi, e);
  return quick_two_sum(p, e);
}

__device__ __forceinline__ dd dd_div(dd x, dd y) {
  const double q1 = __ddiv_rn(x.hi, y.hi);
  dd r = dd_add(x, dd_neg(dd_mul(dd{q1, 0.0}, y)));
  const double q2 = __ddiv_rn(r.hi, y.hi);
  r = dd_add(r, dd_neg(dd_mul(dd{q2, 0.0}, y)));
  const double q3 = __ddiv_rn(r.hi, y.hi);
  dd q = quick_two_sum(q1, q2);
  return dd_add(q, dd{q3, 0.0});
}

// x 2^e for results in the normal range (-1022 <= e <= 1023).
__device__ __forceinline__ double scale2(double x, int e) { return __dmul_rn(x, __hiloint2double((e + 1023) << 20, 0)); }
__device__ __forceinline__ dd dd_scale(dd x, int e) { return dd{scale2(x.hi, e), scale2(x.lo, e)}; }

// 1 / d for d.hi > 0: the double reciprocal and one Newton step, whose
// correction needs only a double.
__device__ __forceinline__ dd dd_inv(dd d) {
  const double r = __drcp_rn(d.hi);
  const double e = __fma_rn(-d.lo, r, __fma_rn(-d.hi, r, 1.0));
  return quick_two_sum(r, __dmul_rn(r, e));
}

// Signed 256-bit integer (w, two's complement) times 2^E as double-double.
// The leading 123 bits form a window whose value is below 2^123, so its
// rounding to double (at most 2^123) converts back to fixed point without
// overflow; hi is that rounding and lo the correctly rounded exact remainder.
// Bits below the window are dropped (relative 2^-122).
__device__ __forceinline__ dd int256_to_dd(const uint64_t *w, int E) {
  uint64_t v0 = w[0], v1 = w[1], v2 = w[2], v3 = w[3];
  const bool neg = (int64_t)v3 < 0;
  if (neg) {
    v0 = ~v0 + 1ull;
    v1 = ~v1 + (v0 == 0 ? 1ull : 0ull);
    v2 = ~v2 + ((v0 | v1) == 0 ? 1ull : 0ull);
    v3 = ~v3 + ((v0 | v1 | v2) == 0 ? 1ull : 0ull);
  }
  const int top = v3 ? 3 : v2 ? 2 : v1 ? 1 : 0;
  const uint64_t vt = v3 ? v3 : v2 ? v2 : v1 ? v1 : v0;
  if (vt == 0) return dd{0.0, 0.0};
  const int L = 64 * top + 63 - __clzll((long long)vt);  // leading bit
  i128 win;
  int Ew = E;
  if (L <= 122) {
    win = mk128(v0, v1);
  } else {
    const int sh = L - 122;  // right shift that puts the leading bit on bit 122
    const int q = sh >> 6, rb = sh & 63;
    const uint64_t a0 = q == 0 ? v0 : q == 1 ? v1 : v2, a1 = q == 0 ? v1 : q == 1 ? v2 : v3,
                   a2 = q == 0 ? v2 : q == 1 ? v3 : 0ull;
    win.lo = rb ? (a0 >> rb) | (a1 << (64 - rb)) : a0;
    win.hi = rb ? (a1 >> rb) | (a2 << (64 - rb)) : a1;
    Ew = E + sh;
  }
  const double hi = fix_to_double(win, Ew).d;
  bool ovf = false;
  const i128 back = double_to_fix(hi, Ew, &ovf);
  const double lo = fix_to_double(add128(win, neg128(back)), Ew).d;
  const dd r{hi, lo};
  return neg ? dd_neg(r) : r;
}

struct FitOut {
  double coef[5];
  double ssr, r2;
  int64_t n;
  int32_t status, dropped;
};

// The status word's bits for the host, and the word cleared for the next call.
__device__ __forceinline__ void hand_status(int *status, int *host) {
  *host = atomicExch(status, 0);
}

// Index of Gram pair (a, b) in the accumulator order (row-major upper triangle).
__host__ __device__ constexpr int gram_idx(int a, int b) {
  return a <= b ? a * 5 - a * (a - 1) / 2 + (b - a) : b * 5 - b * (b - 1) / 2 + (a - b);
}

// Row and column of Gram entry e (inverse of gram_idx: a <= b, row order).
__device__ __forceinline__ void gram_ab(int e, int &a, int &b) {
  a = 0;
  while (e >= 5 - a) {
    e -= 5 - a;
    ++a;
  }
  b = a + e;
}

__device__ __forceinline__ dd dd_sub(dd x, dd y) { return dd_add(x, dd_neg(y)); }

// One block per (y vector k, group g), block k * 4 + g: builds, scales and
// solves the normal equations from the exact totals.  Lanes convert the 21
// totals at once.  The elimination (L D L^T, right-looking, the right-hand side
// as a sixth row) takes one column at a time: every lane inverts the pivot, and
// each of the remaining entries is updated on its own lane, so a column costs
// one inverse, two products and one sum of dependent double-double arithmetic;
// the back substitution and the residual sum go side by side the same way,
// while the second warp forms the total sum of squares.  A dropped a3 column
// becomes a unit row and column with a zero right-hand side (its coefficient
// solves to 0).  Bound by the latency of that chain (one warp, 22 us;
// with a left-looking Cholesky factorisation, one lane on the pivot, 79).  Loops
// stay rolled: the kernel runs once per fit, so its code is fetched cold.
__global__ void __launch_bounds__(64) k_fit_solve(const FitAcc *totals, int n_y, FitOut *__restrict__ out,
                                                   int *status, int *host_status) {
  wait_previous();
  if (blockIdx.x == 0 && threadIdx.x == 0) hand_status(status, host_status);
  __shared__ dd G[15], R[5], A[15], B[5], inv[5];
  __shared__ dd YY, SST;
  __shared__ double cf[5];
  const int tid = threadIdx.x, lane = tid & 31;
  const int k = blockIdx.x / 4, g = blockIdx.x % 4;
  if (k >= n_y) return;
  const int NE = fit_entries(n_y);
  const FitAcc *T = totals + g * NE;
  FitOut o;
  for (int i = 0; i < 5; ++i) o.coef[i] = 0.0;
  o.ssr = 0.0;
  o.r2 = 0.0;
  o.dropped = 0;
  const int64_t n = (int64_t)T[0].w[0];  // Gram (0,0) = number of batches
  o.n = n;
  const bool drop3 = n > 0 && (T[NE - 1].w[0] & 1ull) == 0ull;
  if (drop3) o.dropped = 1 << 3;
  if (n < (drop3 ? 4 : 5)) {
    o.status = LV_ENODATA;
    if (tid == 0) out[k * 4 + g] = o;
    return;
  }
  // exact totals as double-double, one per lane
  if (tid < 21) {
    const int e = tid < 15 ? tid : tid < 20 ? 15 + k * 5 + (tid - 15) : 15 + 5 * n_y + k;
    const dd v = int256_to_dd(T[e].w, tid < 15 ? 0 : tid < 20 ? kFitYLsb : kFitYYLsb);
    if (tid < 15)
      G[tid] = v;
    else if (tid < 20)
      R[tid - 15] = v;
    else
      YY = v;
  }
  __syncthreads();
  if (tid >= 32) {
    if (lane == 0) SST = dd_sub(YY, dd_mul(dd_mul(R[0], R[0]), dd_inv(dd{(double)n, 0.0})));
    __syncthreads();
    return;
  }
  if (drop3 && lane < 5) G[gram_idx(lane, 3)] = dd{lane == 3 ? 1.0 : 0.0, 0.0};
  if (drop3 && lane == 5) R[3] = dd{0.0, 0.0};
  __syncwarp();
  // power-of-two column scaling: scaled diagonal near 1; lane e < 15 holds
  // entry (a, b), a <= b, lane 15 + b the right-hand side of row b
  int a = 5, b = lane - 15;
  if (lane < 15) gram_ab(lane, a, b);
  const bool mine = lane < 20;
  auto scale_of = [&](int c) {
    const int ex = (int)((__double_as_longlong(G[gram_idx(c, c)].hi) >> 52) & 0x7ff) - 1022;  // as frexp gives it
    return -(ex / 2);
  };
  dd v{0.0, 0.0};
  if (mine) v = lane < 15 ? dd_scale(G[lane], scale_of(a) + scale_of(b)) : dd_scale(R[b], scale_of(b));
  if (lane < 15) A[lane] = v;
  if (mine && lane >= 15) B[b] = v;
  __syncwarp();
  bool sing = false;
  for (int j = 0; j < 5; ++j) {
    const dd d = A[gram_idx(j, j)];
    if (!(d.hi > 1e-24)) {
      sing = true;
      break;
    }
    const dd r = dd_inv(d);
    if (lane == 0) inv[j] = r;
    // entry (a, b) of the rest: less l_aj A_bj, l_aj = A_aj / d; a right-hand side: less l_bj B_j
    if (mine && b > j && (lane >= 15 || a > j)) {
      const dd x = lane < 15 ? A[gram_idx(a, j)] : B[j];
      v = dd_sub(v, dd_mul(dd_mul(x, r), A[gram_idx(b, j)]));
    }
    __syncwarp();
    if (lane < 15)
      A[lane] = v;
    else if (mine)
      B[b] = v;
    __syncwarp();
  }
  if (sing) {
    o.status = LV_ESINGULAR;
    if (lane == 0) out[k * 4 + g] = o;
    __syncthreads();
    return;
  }
  // L^T x = D^-1 b, highest index first: lane i holds x_i
  dd x{0.0, 0.0};
  if (lane < 5) x = dd_mul(B[lane], inv[lane]);
  for (int m = 4; m > 0; --m) {
    const dd xm{__shfl_sync(0xffffffffu, x.hi, m), __shfl_sync(0xffffffffu, x.lo, m)};
    if (lane < m) x = dd_sub(x, dd_mul(dd_mul(A[gram_idx(lane, m)], inv[lane]), xm));
  }
  if (lane < 5) cf[lane] = (drop3 && lane == 3) ? 0.0 : scale2(x.hi + x.lo, scale_of(lane));
  __syncwarp();
  for (int i = 0; i < 5; ++i) o.coef[i] = cf[i];
  // residuals of the rounded coefficients: SSR = y'y - 2 c'X'y + c'Gc (unscaled),
  // one term per lane, summed across the warp
  dd term{0.0, 0.0};
  if (lane < 25) {
    const int i = lane / 5, j = lane % 5;
    term = dd_mul(dd_mul(dd{cf[i], 0.0}, dd{cf[j], 0.0}), G[gram_idx(i, j)]);
  } else if (lane < 30) {
    term = dd_neg(dd_scale(dd_mul(dd{cf[lane - 25], 0.0}, R[lane - 25]), 1));
  }
  for (int d = 16; d; d >>= 1)
    term = dd_add(term, dd{__shfl_xor_sync(0xffffffffu, term.hi, d), __shfl_xor_sync(0xffffffffu, term.lo, d)});
  __syncthreads();  // SST
  if (lane == 0) {
    const dd ssr = dd_add(YY, term);
    o.ssr = ssr.hi + ssr.lo;
    const double sstv = SST.hi + SST.lo;
    o.r2 = sstv != 0.0 ? 1.0 - o.ssr / sstv : __longlong_as_double(0x7ff8000000000000ll);
    o.status = LV_OK;
    out[k * 4 + g] = o;
  }
}

}  // namespace lv
