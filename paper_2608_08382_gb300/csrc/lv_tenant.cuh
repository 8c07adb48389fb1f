// Exact per-tenant sums of many shares: the shared-memory table of a CTA and
// the kernel over given shares.
#pragma once

#include "lv_kernels.cuh"

namespace lv {

// Hot tenants (ids below H) in shared memory.  The sum of a tenant's q = share
// * 2^72, modulo 2^128, is four 32-bit words.  Words 0 and 1 have two copies,
// to one of which a lane always adds, so that one tenant's many requests do
// not all serialise in one bank (8 or 32 copies were no faster); words 2 and 3,
// which few additions reach, have one.  Layout, for room of `cap` tenants:
// word 0 [2 cap] and 32 words, one per lane, where lanes with nothing to add do
// so; word 1 the same; word 2 [cap]; word 3 [cap].  Ids from H up add 32-bit
// limbs to the global pending counters.
struct TenTab {
  uint32_t w, sink, w2, w3;  // shared-memory byte addresses: the lane's copy of tenant 0's word 0; its sink; words 2, 3
  uint32_t plane;            // bytes from a word 0 to its word 1
  uint32_t H, n;             // hot tenants, tenants
  unsigned long long *pend;  // [n][4]
};

__host__ __device__ constexpr size_t ten_table_bytes(int cap) { return sizeof(uint32_t) * (size_t)(6 * cap + 64); }

__device__ __forceinline__ TenTab ten_table(const uint32_t *smem, int cap, int H, int n, unsigned long long *pend) {
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem), lane = threadIdx.x & 31u;
  TenTab t;
  t.plane = 4u * (2u * cap + 32u);
  t.w = base + 4u * (lane & 1u);
  t.sink = base + 4u * (2u * cap + lane);
  t.w2 = base + 2u * t.plane;
  t.w3 = t.w2 + 4u * cap;
  t.H = (uint32_t)H;
  t.n = (uint32_t)n;
  t.pend = pend;
  return t;
}

// The table's totals into the pending counters (after a barrier).
__device__ __forceinline__ void ten_table_flush(const uint32_t *smem, int cap, int H, unsigned long long *pend, int tid,
                                                int threads) {
  const int P = 2 * cap + 32;
  for (int u = tid; u < H; u += threads) {
    i128 v = mk128(0ull, (uint64_t)smem[2 * P + u] | ((uint64_t)smem[2 * P + cap + u] << 32));
#pragma unroll
    for (int r = 0; r < 2; ++r)
      v = add128(v, mk128((uint64_t)smem[2 * u + r] | ((uint64_t)smem[P + 2 * u + r] << 32), 0ull));
    if (v.lo | v.hi) pend_add(pend, u, v);
  }
}

// The fold by the last CTA to finish (every CTA calls this once its additions
// to the pending counters are issued): for few tenants one CTA's pass over them
// costs less than a launch of k_tenant_fold.  A call on 6.5e5 requests with and
// without that launch: 16 tenants 22.6 and 21.1 us, 600 44.2 and 42.5, 1,280 34.2
// and 33.8, 2,048 35.6 and 36.9.  (Between the counts the time goes into the cold
// tenants' global atomics, most where a few of them share all of those: 512
// tenants 28 us, 520 34, 600 42, 800 38.)
constexpr int kFoldInline = 1536;
__device__ __forceinline__ void ten_fold_last(unsigned long long *pend, i128 *state, unsigned *ticket, int n,
                                              int *status, int tid, int threads) {
  __shared__ bool last;
  __threadfence();  // this thread's additions before the CTA's ticket
  __syncthreads();
  if (tid == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int u = tid; u < n; u += threads) fold_tenant(pend, state, u, status);
  if (tid == 0) *ticket = 0u;
}

// Shared-memory atomic add at a byte address (address space stated, so that it
// compiles to the shared-memory instruction wherever the table comes from).
__device__ __forceinline__ uint32_t atom_shared(uint32_t addr, uint32_t v) {
  uint32_t o;
  asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(o) : "r"(addr), "r"(v));
  return o;
}

// The carry of x + y.
__device__ __forceinline__ uint32_t carry_of(uint32_t x, uint32_t y) {
  uint32_t c;
  asm("{\n .reg .u32 t;\n add.cc.u32 t, %1, %2;\n addc.u32 %0, 0, 0;\n}" : "=r"(c) : "r"(x), "r"(y));
  return c;
}

// q = (h1:h0) 2^64 + (hi:lo), modulo 2^128, to tenant u < H.  Each word's
// atomic returns its old value, so the lane whose addition wraps a word
// carries into the next: the sum stays exact under any interleaving.
__device__ __forceinline__ void ten_carry(const TenTab &tt, uint32_t u, uint32_t h0, uint32_t h1) {
  if (h0 | h1) {
    h1 += carry_of(atom_shared(tt.w2 + 4u * u, h0), h0);
    if (h1) atom_shared(tt.w3 + 4u * u, h1);
  }
}
__device__ __forceinline__ void ten_add(const TenTab &tt, uint32_t u, uint32_t lo, uint32_t hi, uint32_t h0,
                                        uint32_t h1) {
  const uint32_t w = tt.w + 8u * u;
  const uint32_t c0 = carry_of(atom_shared(w, lo), lo), a1 = hi + c0;
  const uint32_t c1 = carry_of(atom_shared(w + tt.plane, a1), a1) + (a1 < c0 ? 1u : 0u);
  h0 += c1;
  h1 += h0 < c1 ? 1u : 0u;
  ten_carry(tt, u, h0, h1);
}

// Tenant contributions of a lane's four positive normal shares (d: their
// doubles' words) in the common case, a valid tenant and a share in [2^-20, 2^-8
// (1 - 2^-21)) s (then q is whole and below 2^64 - 2^32, so a carry into its
// high word does not wrap); go[k] is cleared otherwise.  The four low words'
// atomics are issued together, then the four high words', so that a lane waits
// for two of them and not for eight; lanes with nothing to add use a word of
// their own, so there is no branch.
constexpr uint32_t kShareLo = (uint32_t)(1075 + kTenLsb) << 20, kShareHi = kShareLo + (12u << 20) - 1u;
__device__ __forceinline__ void ten_add4(const TenTab &tt, bool *go, const uint32_t *u, const uint32_t *dlo,
                                         const uint32_t *dhi) {
  uint32_t w[4], lo[4], hi[4], c1[4];
  bool cold = false;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t sh = (dhi[k] >> 20) - (uint32_t)(1075 + kTenLsb);
    lo[k] = dlo[k] << (sh & 31u);
    hi[k] = __funnelshift_l(dlo[k], (dhi[k] & 0xfffffu) | 0x100000u, sh);
    go[k] = go[k] && dhi[k] - kShareLo < kShareHi - kShareLo && u[k] < tt.n;
    const bool hot = go[k] && u[k] < tt.H;
    w[k] = tt.w + 8u * u[k];
    w[k] = hot ? w[k] : tt.sink;
    cold |= go[k] && !hot;
  }
  if (cold) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (go[k] && u[k] >= tt.H) {
        unsigned long long *pw = tt.pend + 4 * (int64_t)u[k];
        atomicAdd(pw, (unsigned long long)lo[k]);
        atomicAdd(pw + 1, (unsigned long long)hi[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) c1[k] = atom_shared(w[k], lo[k]);
#pragma unroll
  for (int k = 0; k < 4; ++k)  // no wrap
    asm("{\n .reg .u32 t;\n add.cc.u32 t, %1, %2;\n addc.u32 %0, %0, 0;\n}" : "+r"(hi[k]) : "r"(c1[k]), "r"(lo[k]));
#pragma unroll
  for (int k = 0; k < 4; ++k) c1[k] = atom_shared(w[k] + tt.plane, hi[k]);
  uint32_t any = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    c1[k] = carry_of(c1[k], hi[k]);
    any |= c1[k];
  }
  if (any) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (c1[k] && go[k] && u[k] < tt.H) ten_carry(tt, u[k], 1u, 0u);
  }
}

// Any positive normal share with q of at most three words and a valid tenant;
// false otherwise.
__device__ __forceinline__ bool tenant_add_pos(const TenTab &tt, uint32_t u, uint32_t dlo, uint32_t dhi) {
  const uint32_t mh = (dhi & 0xfffffu) | 0x100000u;
  const int sh = (int)(dhi >> 20) - (1075 + kTenLsb);
  if ((unsigned)sh > 42u || u >= tt.n) return false;
  const bool lowp = sh < 32;
  const int t = lowp ? sh : sh - 32;
  const uint32_t x0 = dlo << t, x1 = __funnelshift_l(dlo, mh, t), x2 = t ? mh >> (32 - t) : 0u;
  const uint32_t q0 = lowp ? x0 : 0u, q1 = lowp ? x1 : x0, q2 = lowp ? x2 : x1;
  if (u < tt.H) {
    ten_add(tt, u, q0, q1, q2, 0u);
    return true;
  }
  unsigned long long *pw = tt.pend + 4 * (int64_t)u;
  if (q0) atomicAdd(pw, (unsigned long long)q0);
  if (q1) atomicAdd(pw + 1, (unsigned long long)q1);
  if (q2) atomicAdd(pw + 2, (unsigned long long)q2);
  return true;
}

// The general tenant add (any sign and magnitude; invalid ids are clamped).
__device__ __forceinline__ void tenant_add_any(const TenTab &tt, int32_t u, const Rounded &r, int *bad) {
  if (u < 0 || (uint32_t)u >= tt.n) {
    *bad = 1;
    u = u < 0 ? 0 : (int32_t)tt.n - 1;
  }
  const i128 q = share_to_tenant_fix(r, bad);
  if ((q.lo | q.hi) == 0) return;
  if ((uint32_t)u < tt.H)
    ten_add(tt, (uint32_t)u, (uint32_t)q.lo, (uint32_t)(q.lo >> 32), (uint32_t)q.hi, (uint32_t)(q.hi >> 32));
  else
    pend_add(tt.pend, u, q);
}

// The same, out of line (zero, negative, subnormal or large shares, invalid ids).
__device__ __noinline__ void tenant_add_rare(const TenTab &tt, int32_t u, double d, int *status) {
  int bad = 0;
  tenant_add_any(tt, u, decompose(d), &bad);
  if (bad) flag(status, kStatusData);
}

// Given shares into the accumulator: one CTA per SM, four shares per thread and
// turn, hot tenants in the CTA's table, the table into the pending counters at
// the end.  H: hot tenants (the host makes all of them hot, up to kAccHotMax,
// when there are enough shares that adding the tables costs less than adding
// the cold tenants' shares one by one).  Bound by the atomics' latency and
// throughput, then HBM (12 B a share): 3e7 shares of 3,000 tenants take 80 us,
// 0.66 of the copy rate; 186 with one share per turn, the general add and 512
// hot tenants.
constexpr int kAccThreads = 1024;
constexpr int kAccHotMax = 8192;
__global__ void __launch_bounds__(kAccThreads, 1)
    k_tenant_acc(const double *__restrict__ share, const int32_t *__restrict__ ten, int64_t n,
                 unsigned long long *pend, int32_t n_tenants, int32_t H, int *status, i128 *state, unsigned *ticket) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint32_t *tw = reinterpret_cast<uint32_t *>(smem_raw);
  const TenTab tt = ten_table(tw, H, H, n_tenants, pend);
  for (int i = threadIdx.x; i < (int)(ten_table_bytes(H) / 4); i += kAccThreads) tw[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * (4 * kAccThreads);
  for (int64_t i = blockIdx.x * (int64_t)(4 * kAccThreads) + threadIdx.x; i < n; i += stride) {
    double d[4];
    uint32_t u[4], dlo[4], dhi[4];
    bool in[4], go[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      in[k] = i + k * kAccThreads < n;
      d[k] = in[k] ? __ldcs(share + i + k * kAccThreads) : 0.0;
      u[k] = in[k] ? (uint32_t)__ldcs(ten + i + k * kAccThreads) : 0u;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      dlo[k] = (uint32_t)__double2loint(d[k]);
      dhi[k] = (uint32_t)__double2hiint(d[k]);
      go[k] = in[k] && dhi[k] >= 0x00100000u;  // with ten_add4's bound: positive and normal
    }
    ten_add4(tt, go, u, dlo, dhi);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (in[k] && !go[k]) tenant_add_rare(tt, (int32_t)u[k], d[k], status);
  }
  __syncthreads();
  ten_table_flush(tw, H, H, pend, threadIdx.x, kAccThreads);
  if (state) ten_fold_last(pend, state, ticket, n_tenants, status, threadIdx.x, kAccThreads);
}

}  // namespace lv
