// Consumers of the hyperedge resistances: Algorithm 1 step 6 (sort) and one
// coarsening level of Algorithm 2 (Section III-B, steps 4-10), with Eq.
// R_W_update of Section III-A.3.  Readings of the paper (it fixes neither the
// threshold nor any tie rule), as stated in include/hef.h:
//  - Eq. R_W_update sums eta over a hyperedge's pins in pin order from 0.0,
//    then adds R_e (FP64).
//  - the sort is by ascending updated resistance, ties by ascending id;
//  - delta is given, or the q-quantile (position floor(q (c - 1)) of the c
//    hyperedges with >= 2 pins in sorted order); contraction needs R_e < delta;
//  - contraction is greedy in sorted order: a hyperedge is contracted when
//    none of its pins belongs to an earlier contracted hyperedge;
//  - supernodes are numbered by their smallest vertex, weighted by the
//    resistance of the hyperedge that formed them;
//  - isolated vertices (seeds) join the neighbouring supernode at the smallest
//    distance max_i (Q[p,i] - mu_c[i])^2 / Q_H[i] (mu_c = mean row of the
//    supernode's members, summed in pin order), ties to the smallest id, and
//    add eta(p) + d to its weight in ascending p order;
//  - final ids are compact in the order of each cluster's smallest vertex; the
//    coarse hypergraph keeps each hyperedge's first occurrence of every
//    cluster and drops hyperedges left with fewer than 2 pins.
// Every result is a deterministic function of the inputs: integer atomics
// only, FP64 sums in the stated orders with explicit round-to-nearest
// operations (no contraction into fused multiply-adds), so the results equal
// a sequential CPU statement of the same rules bit for bit.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "internal.h"

namespace hef {

namespace {

#define HEF_PASS(x)              \
  do {                           \
    hef_status s_ = (x);         \
    if (s_ != HEF_OK) return s_; \
  } while (0)

constexpr int kStateLive = 0, kStateIn = 1, kStateOut = 2;
constexpr unsigned int kSpinIters = 1u << 21;  // bounded barrier wait

// FP64 keys as order-preserving unsigned integers (-0.0 taken as +0.0).
__device__ __forceinline__ unsigned long long ordered_bits(double x) {
  unsigned long long b = (unsigned long long)__double_as_longlong(x == 0.0 ? 0.0 : x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Eq. R_W_update per hyperedge (thread per hyperedge, pins in order) and the
// low words of the sort keys.
__global__ void k_update_r(int m, const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
                           const double* __restrict__ R, const double* __restrict__ eta,
                           double* __restrict__ Ru, uint32_t* __restrict__ keys,
                           int32_t* __restrict__ vals) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m) return;
  double acc = 0.0;
  if (eta) {
    for (int64_t t = eptr[e]; t < eptr[e + 1]; ++t) acc = __dadd_rn(acc, eta[pins[t]]);
  }
  const double r = __dadd_rn(acc, R[e]);
  if (Ru) Ru[e] = r;
  keys[e] = (uint32_t)(ordered_bits(r) & 0xffffffffull);
  vals[e] = e;
}

__global__ void k_high_keys(int m, const double* __restrict__ Ru, const int32_t* __restrict__ vals,
                            uint32_t* __restrict__ keys) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) keys[i] = (uint32_t)(ordered_bits(Ru[vals[i]]) >> 32);
}

// rank[order[i]] = i; flags of the hyperedges with >= 2 pins in sorted order.
__global__ void k_rank(int m, const int32_t* __restrict__ order, const int64_t* __restrict__ eptr,
                       int32_t* __restrict__ rank, int* __restrict__ big) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int e = order[i];
  rank[e] = i;
  big[i] = (eptr[e + 1] - eptr[e]) >= 2 ? 1 : 0;
}

// delta: the given value, or the q-quantile of the resistances of the
// hyperedges with >= 2 pins (pos = their exclusive scan in sorted order).
__global__ void k_delta(int m, double given, double q, const int32_t* __restrict__ order,
                        const double* __restrict__ Ru, const int* __restrict__ big,
                        const int* __restrict__ pos, double* __restrict__ delta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (given >= 0.0) {
    if (i == 0) *delta = given;
    return;
  }
  const int c = pos[m];
  if (c == 0) {
    if (i == 0) *delta = INFINITY;
    return;
  }
  const int want = (int)floor(__dmul_rn(q, (double)(c - 1)));
  if (i < m && big[i] && pos[i] == want) *delta = Ru[order[i]];
}

__global__ void k_contract_init(int n, int m, const int64_t* __restrict__ eptr,
                                const double* __restrict__ Ru, const double* __restrict__ delta,
                                int* __restrict__ state, int* __restrict__ best,
                                int32_t* __restrict__ owner) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const double d = *delta;
  if (i < m) state[i] = ((eptr[i + 1] - eptr[i]) >= 2 && Ru[i] < d) ? kStateLive : kStateOut;
  if (i < n) best[i] = 0x7fffffff, owner[i] = -1;
}

// Grid barrier of the contraction kernel: arrivals on a monotonic counter,
// bounded wait.  Returns false when the wait ran out (status set).
__device__ __forceinline__ bool grid_sync(unsigned int* count, unsigned int target,
                                          int* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    unsigned int it = 0;
    int good = 1;
    while (*reinterpret_cast<volatile unsigned int*>(count) < target) {
      if (++it > kSpinIters || *reinterpret_cast<volatile int*>(status)) {
        atomicOr(status, 1);
        good = 0;
        break;
      }
    }
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok;
}

// The greedy contraction as rounds (one cooperative launch): in each round a
// live candidate whose rank is the smallest among the live candidates at
// every one of its pins is contracted (such hyperedges are pin-disjoint),
// and a live candidate with a pin taken by a contracted hyperedge drops out.
// A live candidate is contracted exactly when every earlier candidate that
// shares a pin with it has dropped out, which is the sequential greedy rule;
// every round decides at least the smallest live rank, so at most
// (candidates + 1) rounds run.  round_live[r] counts the live candidates left
// after round r.
__global__ void k_contract(int m, const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
                           const int32_t* __restrict__ rank, int* state, int* best, int32_t* owner,
                           int* last, int* round_live, unsigned int* count, int* status) {
  const int stride = gridDim.x * blockDim.x;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned int ph = 0;
  for (int r = 0; r <= m; ++r) {
    // 1: every live candidate marks its rank at its pins
    for (int e = tid; e < m; e += stride) {
      if (__ldcg(state + e) != kStateLive) continue;
      last[e] = r;
      const int rk = rank[e];
      for (int64_t t = eptr[e]; t < eptr[e + 1]; ++t) atomicMin(best + pins[t], rk);
    }
    if (!grid_sync(count, (++ph) * gridDim.x, status)) return;
    // 2: the smallest live rank at all of its pins is contracted
    for (int e = tid; e < m; e += stride) {
      if (__ldcg(state + e) != kStateLive) continue;
      const int rk = rank[e];
      bool mine = true;
      for (int64_t t = eptr[e]; t < eptr[e + 1] && mine; ++t) mine = __ldcg(best + pins[t]) == rk;
      if (mine) {
        state[e] = kStateIn;
        for (int64_t t = eptr[e]; t < eptr[e + 1]; ++t) owner[pins[t]] = e;
      }
    }
    if (!grid_sync(count, (++ph) * gridDim.x, status)) return;
    // 3: live candidates with a taken pin drop out; the round's marks are cleared
    for (int e = tid; e < m; e += stride) {
      if (__ldcg(last + e) != r) continue;
      const int st = __ldcg(state + e);
      bool taken = false;
      for (int64_t t = eptr[e]; t < eptr[e + 1]; ++t) {
        best[pins[t]] = 0x7fffffff;
        taken = taken || __ldcg(owner + pins[t]) >= 0;
      }
      if (st == kStateLive) {
        if (taken) state[e] = kStateOut;
        else atomicAdd(round_live + r, 1);
      }
    }
    if (!grid_sync(count, (++ph) * gridDim.x, status)) return;
    if (__ldcg(round_live + r) == 0) return;
  }
  if (threadIdx.x == 0 && blockIdx.x == 0) atomicOr(status, 2);  // more rounds than possible
}

// Smallest pin of every contracted hyperedge.
__global__ void k_minpin(int m, const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
                         const int* __restrict__ state, int32_t* __restrict__ minpin) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m || state[e] != kStateIn) return;
  int mn = 0x7fffffff;
  for (int64_t t = eptr[e]; t < eptr[e + 1]; ++t) mn = min(mn, pins[t]);
  minpin[e] = mn;
}

__global__ void k_cluster_flags(int n, const int32_t* __restrict__ owner,
                                const int32_t* __restrict__ minpin, int* __restrict__ flag) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int o = owner[v];
  flag[v] = (o < 0 || minpin[o] == v) ? 1 : 0;
}

__global__ void k_clusters(int n, const int32_t* __restrict__ owner, const int32_t* __restrict__ minpin,
                           const int* __restrict__ cid, const double* __restrict__ Ru,
                           const double* __restrict__ eta, int32_t* __restrict__ cluster,
                           double* __restrict__ eta_next, int32_t* __restrict__ formed_by,
                           int* __restrict__ contracted_flag) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int o = owner[v];
  const int c = o < 0 ? cid[v] : cid[minpin[o]];
  cluster[v] = c;
  if (o < 0) {
    eta_next[c] = eta ? eta[v] : 0.0;
    formed_by[c] = -1;
    contracted_flag[c] = 0;
  } else if (minpin[o] == v) {
    eta_next[c] = Ru[o];
    formed_by[c] = o;
    contracted_flag[c] = 1;
  }
}

// (double)x by integer operations for normal x: conversions to FP64 share the
// FP64 pipe's rate of two per clock and SM.
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return (double)x;  // zero, subnormal, infinite, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

template <typename T>
__device__ __forceinline__ double qval(const T* Q, long long ldq, long long row, int i) {
  if constexpr (std::is_same<T, __nv_bfloat16>::value) return widen(__bfloat162float(Q[row * ldq + i]));
  else if constexpr (std::is_same<T, float>::value) return widen(Q[row * ldq + i]);
  else return Q[row * ldq + i];
}

// a / k rounded to nearest (as __ddiv_rn) for an integer 2 <= k < 2^31 given
// with rk = 1/k rounded to nearest: q0 is within two ulps, its residual is
// exact, and the corrected quotient is off by less than 2^-104 of itself before
// its rounding, while a quotient by k that is no rounding boundary lies at
// least 2^-54 / k away from one.  Three FP64 operations (one when k is a power
// of two) instead of a division's sequence and its special cases; tiny and
// non-finite values take the division.
__device__ __forceinline__ double div_by_int(double a, double k, double rk, bool pow2) {
  const int f = (__double2hiint(a) >> 20) & 0x7ff;
  if (f < 200 || f > 2000) return __ddiv_rn(a, k);
  const double q0 = __dmul_rn(a, rk);
  if (pow2) return q0;
  return __fma_rn(__fma_rn(-k, q0, a), rk, q0);
}

// x truncated to FP32 (rounded where its exponent is out of the normal range).
__device__ __forceinline__ float narrow(double x) {
  const unsigned h = (unsigned)__double2hiint(x), f = (h >> 20) & 0x7ffu;
  if (f < 897u || f > 1150u) return (float)x;
  return __uint_as_float((h & 0x80000000u) | ((((h & 0x7fffffffu) - (896u << 20)) << 3) |
                                              ((unsigned)__double2loint(x) >> 29)));
}

// Centroid rows of the contracted supernodes: one warp per supernode, NC
// columns per lane, members summed in the forming hyperedge's pin order (one
// round of row loads per member).  Also what k_seeds reads: the FP32 rows mu32;
// the column scales scale[i] = 1/Q_H[i] (0 for columns that take no part),
// scale[K] = 1 when some Q_H lies outside [1e-30, 1e30], where FP32 bounds could
// overflow or underflow and every distance is formed in FP64; and for every
// vertex its supernode and that supernode's row, or -1 when it is isolated.
// Bound by the FP64 pipe (one add per member and column, then the division):
// 186 -> 152 us at 210,000 vertices, K = 160.
template <typename T, int NC>
__global__ void __launch_bounds__(kThreads)
    k_centroids(int n, const int32_t* __restrict__ formed_by, const int* __restrict__ mrow,
                const int32_t* __restrict__ cluster, const int64_t* __restrict__ eptr,
                const int32_t* __restrict__ pins, const T* __restrict__ Q, long long ldq, int K,
                const double* __restrict__ QH, double* __restrict__ mu, float* __restrict__ mu32,
                float* __restrict__ scale, int2* __restrict__ vinfo) {
  if (blockIdx.x == 0) {
    int wide = 0;
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
      const double h = QH[i];
      const bool on = h > 1e-300;
      wide |= on && !(h >= 1e-30 && h <= 1e30);
      scale[i] = on ? (float)(1.0 / h) : 0.0f;
    }
    wide = __syncthreads_or(wide);
    if (threadIdx.x == 0) scale[K] = wide ? 1.0f : 0.0f;
  }
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid < n) {
    const int cv = cluster[tid];
    vinfo[tid] = formed_by[cv] >= 0 ? make_int2(cv, mrow[cv]) : make_int2(-1, 0);
  }
  const int lane = threadIdx.x & 31;
  const int c = (int)(tid >> 5);
  if (c >= n) return;
  const int e = formed_by[c];
  if (e < 0) return;
  const int64_t a = eptr[e], b = eptr[e + 1];
  const double k = (double)(b - a), rk = __ddiv_rn(1.0, k);
  const bool pow2 = ((b - a) & (b - a - 1)) == 0;
  double acc[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) acc[j] = 0.0;
  for (int64_t t = a; t < b; ++t) {
    const int u = pins[t];
    double x[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) x[j] = lane + 32 * j < K ? qval(Q, ldq, u, lane + 32 * j) : 0.0;
#pragma unroll
    for (int j = 0; j < NC; ++j)
      if (32 * j < K) acc[j] = __dadd_rn(acc[j], x[j]);  // no FP64 for absent columns
  }
  const size_t row = (size_t)mrow[c] * K;
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const int i = lane + 32 * j;
    if (i < K) {
      const double x = div_by_int(acc[j], k, rk, pow2);
      mu[row + i] = x;
      mu32[row + i] = narrow(x);
    }
  }
}

// Local clustering of the isolated vertices: one warp per vertex; every
// candidate supernode (of a co-pin in a hyperedge containing the vertex) is
// scored by max over columns of (Q[p,i] - mu_c[i])^2 / Q_H[i]; the smallest
// score wins, ties to the smallest cluster id.
//
// The scores are FP64 (round to nearest), and FP64 division would bound this
// kernel (two DFMA per clock and SM): with K divisions per candidate pin it takes
// 5.68 ms at 210,000 vertices, K = 160, as it is 0.46 ms.  A candidate is bounded
// in FP32 first: with
// q, m the FP32 values of Q[p,i] and mu_c[i] (rounded and truncated), |Q - mu|
// lies within err = 1.5 2^-23 (|q| + |m|) of |q - m|, which gives [lb_i, ub_i] around each
// column's ratio and [max lb, max ub] around the score (the constants below
// leave slack for every rounding, underflow included).  A candidate whose lower
// bound exceeds an earlier candidate's upper bound cannot win; for the others
// only the columns with ub_i >= max lb can hold the maximum, and only those
// are formed in FP64: one or two divisions for a few candidates per vertex,
// with the same result bit for bit.  Columns are held NC per lane, so a
// candidate costs one FP32 row of gathers.  What remains is the chain of
// dependent loads from a vertex to its candidates' rows: the lanes take the pins
// of up to 32 hyperedges together, 32 pins at a time, which walks it once for
// most vertices instead of once per hyperedge.
// CTAs of two warps: a CTA keeps its registers until its slowest vertex is done,
// and about half the vertices have nothing to do.
constexpr int kSeedThreads = 64;

template <typename T, int NC>
__global__ void __launch_bounds__(kSeedThreads)
    k_seeds(int n, const int32_t* __restrict__ owner, const int32_t* __restrict__ vptr,
            const int32_t* __restrict__ vedge, const int32_t* __restrict__ perm,
            const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
            const int2* __restrict__ vinfo, const double* __restrict__ mu,
            const float* __restrict__ mu32, const float* __restrict__ scale,
            const T* __restrict__ Q, long long ldq, int K, const double* __restrict__ QH,
            int32_t* __restrict__ target, double* __restrict__ dist) {
  constexpr float kErr = 1.9e-7f;       // > 1.5 2^-23
  constexpr float kSlack = 1e-6f;       // relative, > the products' and scales' roundings
  constexpr float kTiny = 1e-37f;       // absolute, > what underflow loses
  const int lane = threadIdx.x & 31;
  const int p = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (p >= n) return;
  if (owner[p] >= 0) {
    if (lane == 0) target[p] = -1, dist[p] = 0.0;
    return;
  }
  const bool wide = scale[K] != 0.0f;
  float q[NC], sc[NC];
#pragma unroll
  for (int t = 0; t < NC; ++t) {
    const int i = lane + 32 * t;
    q[t] = i < K ? (float)qval(Q, ldq, p, i) : 0.0f;
    sc[t] = i < K ? scale[i] : 0.0f;
  }
  int best = -1;
  double bd = INFINITY;
  float bound = INFINITY;  // smallest upper bound of a candidate so far
  const int t1 = vptr[p + 1];
  for (int t0 = vptr[p]; t0 < t1; t0 += 32) {
    // lane l: the pins [first, first + cnt) of hyperedge t0 + l, at [at, at +
    // cnt) of the round's pins
    int64_t first = 0;
    int cnt = 0;
    if (t0 + lane < t1) {
      const int e = perm[vedge[t0 + lane]];
      first = eptr[e];
      cnt = (int)(eptr[e + 1] - first);
    }
    int end = cnt;  // inclusive sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += x;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    const int at = end - cnt;
    for (int s0 = 0; s0 < total; s0 += 32) {
      // pin s0 + lane lies in the hyperedge of the last lane whose start is at
      // or before it (empty hyperedges share their successor's start)
      int h = 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        if (__shfl_sync(0xffffffffu, at, h + o) <= s0 + lane) h += o;
      const int64_t hf = __shfl_sync(0xffffffffu, (long long)first, h);
      const int ha = __shfl_sync(0xffffffffu, at, h);
      int c = -1 - lane, row = 0;
      if (s0 + lane < total) {
        const int u = pins[hf + (s0 + lane - ha)];
        const int2 v = vinfo[u];
        if (u != p && v.x >= 0) c = v.x, row = v.y;
      }
      // each supernode once per 32 pins
      const unsigned peers = __match_any_sync(0xffffffffu, c);
      unsigned todo = __ballot_sync(0xffffffffu, c >= 0 && lane == __ffs(peers) - 1);
      // bounds of every candidate first, kept by its lane; then FP64 for those
      // that the smallest upper bound leaves (a warp's FP64 operation takes 16
      // cycles of the SM's pipe however few of its lanes are on)
      auto bounds = [&](size_t ro, float (&ub)[NC], float& lo, float& hi) {
        float m[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) m[j] = lane + 32 * j < K ? mu32[ro + lane + 32 * j] : 0.0f;
        lo = 0.0f, hi = 0.0f;
        bool open = false;  // overflow or NaN: no upper bound
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          if (32 * j < K) {
            const float d = fabsf(q[j] - m[j]), size = fabsf(q[j]) + fabsf(m[j]);
            const float du = fmaf(kErr, size, d), dl = fmaxf(fmaf(-kErr, size, d), 0.0f);
            ub[j] = du * sc[j] * du;
            open |= !(ub[j] <= 3.0e38f);
            hi = fmaxf(hi, ub[j]);
            lo = fmaxf(lo, dl * sc[j] * dl);
          }
        }
        // non-negative floats order as their bits
        hi = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(open ? INFINITY : hi)));
        lo = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(lo)));
        hi = hi * (1.0f + kSlack) + kTiny;
        lo = fmaxf(fminf(lo, 3.0e38f) * (1.0f - kSlack) - kTiny, 0.0f);
        if (wide) lo = 0.0f, hi = INFINITY;
      };
      float ub[NC], lo, hi, mylo = INFINITY;
      for (unsigned rest = todo; rest; rest &= rest - 1) {
        const int src = __ffs(rest) - 1;
        bounds((size_t)__shfl_sync(0xffffffffu, row, src) * K, ub, lo, hi);
        if (lane == src) mylo = lo;
        bound = fminf(bound, hi);
      }
      todo = __ballot_sync(0xffffffffu, ((todo >> lane) & 1u) && mylo <= bound);
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int cc = __shfl_sync(0xffffffffu, c, src);
        const size_t ro = (size_t)__shfl_sync(0xffffffffu, row, src) * K;
        bounds(ro, ub, lo, hi);
        double d = 0.0;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
          const int i = lane + 32 * j;
          if (i < K && (wide || !(ub[j] * (1.0f + kSlack) + kTiny < lo))) {
            const double qh = QH[i];
            if (qh > 1e-300) {
              const double diff = __dsub_rn(qval(Q, ldq, p, i), mu[ro + i]);
              const double r = __ddiv_rn(__dmul_rn(diff, diff), qh);
              d = r > d ? r : d;
            }
          }
        }
        // the largest of the lanes' non-negative doubles, by their bits
        const unsigned dh = (unsigned)__double2hiint(d), mh = __reduce_max_sync(0xffffffffu, dh);
        const unsigned ml = __reduce_max_sync(0xffffffffu, dh == mh ? (unsigned)__double2loint(d) : 0u);
        d = __hiloint2double((int)mh, (int)ml);
        if (d < bd || (d == bd && cc < best)) best = cc, bd = d;
      }
    }
  }
  if (lane == 0) {
    target[p] = best;
    dist[p] = best >= 0 ? bd : 0.0;
  }
}

// Sort keys of the merges: target + 1 for seeds that join, 0 otherwise.
__global__ void k_merge_keys(int n, const int32_t* __restrict__ target, uint32_t* __restrict__ keys,
                             int32_t* __restrict__ vals) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  keys[v] = (uint32_t)(target[v] + 1);
  vals[v] = v;
}

// Weight of each supernode that seeds join: its own weight, then eta(p) +
// d(p) for the seeds in ascending p (a sorted segment, summed by one thread).
__global__ void k_merge_sums(int n, const uint32_t* __restrict__ keys, const int32_t* __restrict__ vals,
                             const double* __restrict__ eta, const double* __restrict__ dist,
                             double* __restrict__ eta2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || keys[i] == 0u || (i > 0 && keys[i - 1] == keys[i])) return;
  const int c = (int)keys[i] - 1;
  double acc = eta2[c];
  for (int j = i; j < n && keys[j] == keys[i]; ++j) {
    const int p = vals[j];
    acc = __dadd_rn(acc, __dadd_rn(eta ? eta[p] : 0.0, dist[p]));
  }
  eta2[c] = acc;
}

__global__ void k_final_min(int n, const int32_t* __restrict__ cluster, const int32_t* __restrict__ target,
                            int* __restrict__ minv) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int c = target[v] >= 0 ? target[v] : cluster[v];
  atomicMin(minv + c, v);
}

__global__ void k_final_flags(int n, const int32_t* __restrict__ cluster,
                              const int32_t* __restrict__ target, const int* __restrict__ minv,
                              int* __restrict__ flag) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int c = target[v] >= 0 ? target[v] : cluster[v];
  flag[v] = minv[c] == v ? 1 : 0;
}

__global__ void k_final_ids(int n, const int32_t* __restrict__ cluster, const int32_t* __restrict__ target,
                            const int* __restrict__ minv, const int* __restrict__ fid,
                            const double* __restrict__ eta2, int32_t* __restrict__ final_id,
                            double* __restrict__ eta_out) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  const int c = target[v] >= 0 ? target[v] : cluster[v];
  const int f = fid[minv[c]];
  final_id[v] = f;
  if (minv[c] == v) eta_out[f] = eta2[c];
}

// Distinct clusters of a hyperedge, first occurrences in pin order: with
// `out`, written there; returns their count.  A thread per hyperedge that
// compares every pin with all earlier ones is as slow as the longest hyperedge
// (a 400-pin net makes 80,000 dependent two-step gathers).  Here a lane keeps up
// to kRegPins clusters in registers, which covers 96 % of a netlist's
// hyperedges, and longer ones are taken by their warp, 32 pins at a time: equal
// clusters within a round meet by a warp match, earlier rounds by a hash table
// in shared memory, so that the work is linear in the pins.  Hyperedges too long
// for the table compare their rounds with all earlier ones from registers
// instead.  Both kernels are then bound by the two gathers per pin: 2747 -> 23 us
// (fill) and 2736 -> 21 us (count) at 200,000 nets.
constexpr int kRegPins = 8;
constexpr int kHashSlots = 1024;             // per warp; at most half full
constexpr int kHashPins = kHashSlots / 2;    // longer hyperedges skip the table
constexpr int kCoarseWarps = kThreads / 32;

__device__ __forceinline__ int distinct_in_lane(const int32_t* __restrict__ pins, int64_t a, int k,
                                                const int32_t* __restrict__ fid, int32_t* out) {
  int c[kRegPins];
#pragma unroll
  for (int j = 0; j < kRegPins; ++j) c[j] = j < k ? pins[a + j] : 0;
#pragma unroll
  for (int j = 0; j < kRegPins; ++j) c[j] = j < k ? fid[c[j]] : -1;
  int cnt = 0;
#pragma unroll
  for (int j = 0; j < kRegPins; ++j) {
    bool fresh = j < k;
#pragma unroll
    for (int i = 0; i < j; ++i) fresh = fresh && c[i] != c[j];
    if (fresh) {
      if (out) out[cnt] = c[j];
      ++cnt;
    }
  }
  return cnt;
}

// By the whole warp (all arguments warp-uniform); `table` holds kHashSlots ints.
__device__ int distinct_in_warp(const int32_t* __restrict__ pins, int64_t a, int64_t b,
                                const int32_t* __restrict__ fid, int32_t* out, int* table) {
  const int lane = threadIdx.x & 31;
  const int64_t k = b - a;
  const bool hashed = k > 32 && k <= kHashPins;
  if (hashed) {
    for (int i = lane; i < kHashSlots; i += 32) table[i] = -1;
    __syncwarp();
  }
  int cnt = 0;
  for (int64_t t0 = a; t0 < b; t0 += 32) {
    const bool act = t0 + lane < b;
    const int c = act ? fid[pins[t0 + lane]] : -1 - lane;  // inactive lanes match nobody
    const unsigned peers = __match_any_sync(0xffffffffu, c);
    bool fresh = act && lane == __ffs(peers) - 1;
    if (hashed) {
      if (fresh) {
        unsigned h = ((unsigned)c * 2654435761u) >> 22;  // top 10 bits: [0, kHashSlots)
        while (true) {
          const int old = atomicCAS(table + h, -1, c);
          if (old == -1) break;
          if (old == c) {
            fresh = false;
            break;
          }
          h = (h + 1) & (kHashSlots - 1);
        }
      }
      __syncwarp();
    } else {
      for (int64_t u0 = a; u0 < t0; u0 += 32) {  // earlier rounds are full
        const int x = fid[pins[u0 + lane]];
#pragma unroll 8
        for (int q = 0; q < 32; ++q) {
          const int other = __shfl_sync(0xffffffffu, x, q);  // by every lane, fresh or not
          fresh = fresh && other != c;
        }
      }
    }
    const unsigned won = __ballot_sync(0xffffffffu, fresh);
    if (out && fresh) out[cnt + __popc(won & ((1u << lane) - 1u))] = c;
    cnt += __popc(won);
  }
  __syncwarp();  // the table is free for the warp's next hyperedge
  return cnt;
}

// Every lane's own hyperedge [a, b) (empty for lanes without one): its count,
// written to out + off when `out` is given.
__device__ __forceinline__ int distinct_clusters(const int32_t* __restrict__ pins, int64_t a,
                                                 int64_t b, const int32_t* __restrict__ fid,
                                                 int32_t* out, int off) {
  static_assert(kHashSlots == 1 << 10, "the hash keeps 10 bits");
  __shared__ int tables[kCoarseWarps][kHashSlots];
  const int lane = threadIdx.x & 31;
  int cnt = 0;
  const bool in_lane = b - a <= kRegPins;
  if (in_lane) cnt = distinct_in_lane(pins, a, (int)(b - a), fid, out ? out + off : nullptr);
  unsigned todo = __ballot_sync(0xffffffffu, !in_lane);
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int64_t wa = __shfl_sync(0xffffffffu, (long long)a, src);
    const int64_t wb = __shfl_sync(0xffffffffu, (long long)b, src);
    const int wo = __shfl_sync(0xffffffffu, off, src);
    const int c = distinct_in_warp(pins, wa, wb, fid, out ? out + wo : nullptr,
                                   tables[threadIdx.x >> 5]);
    if (lane == src) cnt = c;
  }
  return cnt;
}

__global__ void k_coarse_count(int m, const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
                               const int32_t* __restrict__ fid, int* __restrict__ keep,
                               int* __restrict__ cnt) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = e < m;  // every lane of a warp takes part in its long hyperedges
  const int64_t a = act ? eptr[e] : 0, b = act ? eptr[e + 1] : 0;
  const int k = distinct_clusters(pins, a, b, fid, nullptr, 0);
  if (!act) return;
  keep[e] = k >= 2 ? 1 : 0;
  cnt[e] = k >= 2 ? k : 0;
}

__global__ void k_coarse_fill(int m, const int64_t* __restrict__ eptr, const int32_t* __restrict__ pins,
                              const double* __restrict__ w, const int32_t* __restrict__ fid,
                              const int* __restrict__ keep, const int* __restrict__ ne,
                              const int* __restrict__ po, int64_t* __restrict__ ceptr,
                              int32_t* __restrict__ cpins, double* __restrict__ cw,
                              int32_t* __restrict__ emap) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = e < m && keep[e];
  if (e == m) ceptr[ne[m]] = po[m];
  int off = 0;
  if (act) {
    const int i = ne[e];
    off = po[e];
    ceptr[i] = off;
    cw[i] = w[e];
    emap[i] = e;
  }
  const int64_t a = act ? eptr[e] : 0, b = act ? eptr[e + 1] : 0;
  distinct_clusters(pins, a, b, fid, cpins, off);
}

__global__ void k_counts(const int* __restrict__ nc, const int* __restrict__ nf,
                         const int* __restrict__ mc, const int* __restrict__ pc,
                         const int* __restrict__ status, int32_t* __restrict__ counts) {
  if (threadIdx.x == 0 && blockIdx.x == 0)
    counts[0] = *nc, counts[1] = *nf, counts[2] = *mc, counts[3] = *pc, counts[4] = *status;
}

inline int grid_of(long long N) { return (int)((N + kThreads - 1) / kThreads); }

struct LevelWs {
  uint32_t* keys;
  int32_t* vals;
  SortBufs sb;
  unsigned int* counter;  // [0] scans and sorts, [1] contraction barrier
  int* status;            // [0] contraction wait / round overflow
  int32_t* rank;
  int* state;
  int* last;
  int* round_live;
  int* best;
  int32_t* minpin;
  int* flag;     // max(n, m) + 1
  int* scan;     // max(n, m) + 1
  int* bsum;
  int* cflag;    // n + 1: contracted-cluster flags, scanned into row indices
  int32_t* formed_by;
  double* eta_next;
  double* eta2;
  double* mu;
  int2* vinfo;   // n: supernode and its centroid row, or -1
  float* mu32;   // FP32 rows of mu, scale (K + 1): bounds of the seeds' distances
  float* scale;
  int* minv;
  int* keep;     // m + 1
  int* ne;       // m + 1
  int* po;       // m + 1
};

size_t carve_level(void* base, long long n, long long m, int K, LevelWs* w) {
  Carver c(base);
  const long long N = (n > m ? n : m) + 1;
  w->keys = c.take<uint32_t>(N);
  w->vals = c.take<int32_t>(N);
  carve_sort_bufs(c, N, &w->sb);
  w->counter = c.take<unsigned int>(4);
  w->sb.counter = w->counter;
  w->status = c.take<int>(2);
  w->rank = c.take<int32_t>(m + 1);
  w->state = c.take<int>(m + 1);
  w->last = c.take<int>(m + 1);
  w->round_live = c.take<int>(m + 2);
  w->best = c.take<int>(n + 1);
  w->minpin = c.take<int32_t>(m + 1);
  w->flag = c.take<int>(N + 1);
  w->scan = c.take<int>(N + 1);
  w->bsum = c.take<int>(scan_tiles(N + 1) + 1);
  w->cflag = c.take<int>(n + 1);
  w->formed_by = c.take<int32_t>(n + 1);
  w->eta_next = c.take<double>(n + 1);
  w->eta2 = c.take<double>(n + 1);
  w->mu = c.take<double>((size_t)(n / 2 + 1) * (K > 0 ? K : 1));
  w->mu32 = c.take<float>((size_t)(n / 2 + 1) * (K > 0 ? K : 1));
  w->scale = c.take<float>(K + 1);
  w->vinfo = c.take<int2>(K > 0 ? n + 1 : 1);
  w->minv = c.take<int>(n + 1);
  w->keep = c.take<int>(m + 1);
  w->ne = c.take<int>(m + 1);
  w->po = c.take<int>(m + 1);
  return c.bytes();
}

// Sorted order of R (ascending, ties by id) into `order`: a stable sort on the
// low key words, then on the high words.
hef_status sort_by_value(int m, const double* Ru, int32_t* order, LevelWs& w, cudaStream_t st) {
  if (m <= 0) return HEF_OK;
  HEF_PASS(radix_sort(w.keys, w.vals, m, 32, w.sb, st));
  HEF_LAUNCH("k_high_keys", st, k_high_keys<<<grid_of(m), kThreads, 0, st>>>(m, Ru, w.vals, w.keys));
  HEF_CHECK_LAUNCH();
  HEF_PASS(radix_sort(w.keys, w.vals, m, 32, w.sb, st));
  HEF_CHECK_CUDA(cudaMemcpyAsync(order, w.vals, (size_t)m * sizeof(int32_t),
                                 cudaMemcpyDeviceToDevice, st));
  return HEF_OK;
}

}  // namespace

}  // namespace hef

using namespace hef;

extern "C" size_t hef_level_workspace_bytes(int64_t n, int64_t m, int32_t K) {
  if (n < 0 || m < 0 || K < 0 || K > 512) return 0;
  LevelWs w;
  return carve_level(nullptr, n, m, K, &w);
}

extern "C" hef_status hef_sort_resistance(int64_t m, const double* R, int32_t* order,
                                          void* workspace, size_t workspace_bytes, void* stream) {
  HEF_NVTX("hef_sort_resistance (Algorithm 1 step 6)");
  if (m < 0 || m > 0x7fffffffll) return set_error(HEF_ERR_INVALID_ARG, "hef_sort_resistance: bad m");
  if (m > 0 && (!R || !order)) return set_error(HEF_ERR_INVALID_ARG, "hef_sort_resistance: NULL array");
  LevelWs w;
  const size_t need = carve_level(workspace, 0, m, 0, &w);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need)
    return set_error(HEF_ERR_WORKSPACE, "hef_sort_resistance: workspace needs %zu bytes", need);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (m == 0) return HEF_OK;
  HEF_CHECK_CUDA(cudaMemsetAsync(w.counter, 0, 4 * sizeof(unsigned int), st));
  // keys of R itself (no eta): Eq. R_W_update with eta = 0 is R
  HEF_LAUNCH("k_update_r", st, k_update_r<<<grid_of(m), kThreads, 0, st>>>(
                                   (int)m, nullptr, nullptr, R, nullptr, nullptr, w.keys, w.vals));
  HEF_CHECK_LAUNCH();
  return sort_by_value((int)m, R, order, w, st);
}

extern "C" hef_status hef_coarsen_level(const hef_incidence* inc, const int64_t* eptr,
                                        const int32_t* pins, const double* w, const double* R,
                                        const double* eta, const void* Q, int64_t ldq, int32_t K,
                                        int32_t dtype, const double* QH, double delta,
                                        double quantile, const hef_level_out* out,
                                        void* workspace, size_t workspace_bytes, void* stream) {
  HEF_NVTX("hef_coarsen_level (Algorithm 2 steps 4-10)");
  if (!inc || !out) return set_error(HEF_ERR_INVALID_ARG, "hef_coarsen_level: NULL incidence or out");
  const long long n = inc->n, m = inc->m;
  if (m > 0 && (!eptr || !pins || !w || !R))
    return set_error(HEF_ERR_INVALID_ARG, "hef_coarsen_level: NULL input array");
  if (!out->R_upd || !out->order || !out->delta || !out->owner || !out->cluster || !out->target ||
      !out->dist || !out->final_cluster || !out->eta_out || !out->counts || !out->ceptr ||
      !out->cpins || !out->cw || !out->emap)
    return set_error(HEF_ERR_INVALID_ARG, "hef_coarsen_level: NULL output array");
  if (Q) {
    if (K < 1 || K > 512 || ldq < K || !QH)
      return set_error(HEF_ERR_INVALID_ARG, "hef_coarsen_level: need 1 <= K <= 512, ldq >= K and QH");
    if (dtype != HEF_F64 && dtype != HEF_F32 && dtype != HEF_BF16)
      return set_error(HEF_ERR_INVALID_ARG,
                       "hef_coarsen_level: dtype must be HEF_F64, HEF_F32 or HEF_BF16");
  }
  if (!(delta >= 0.0) && !(quantile >= 0.0 && quantile <= 1.0))
    return set_error(HEF_ERR_INVALID_ARG,
                     "hef_coarsen_level: give delta >= 0, or delta < 0 and 0 <= quantile <= 1");
  LevelWs ws;
  const size_t need = carve_level(workspace, n, m, Q ? K : 0, &ws);
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255) || workspace_bytes < need)
    return set_error(HEF_ERR_WORKSPACE, "hef_coarsen_level: workspace needs %zu bytes", need);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nn = (int)n, mm = (int)m;
  const long long N = (n > m ? n : m);
  HEF_CHECK_CUDA(cudaMemsetAsync(ws.counter, 0, 4 * sizeof(unsigned int), st));
  HEF_CHECK_CUDA(cudaMemsetAsync(ws.status, 0, 2 * sizeof(int), st));
  HEF_CHECK_CUDA(cudaMemsetAsync(ws.round_live, 0, (m + 2) * sizeof(int), st));
  HEF_CHECK_CUDA(cudaMemsetAsync(out->counts, 0, 5 * sizeof(int32_t), st));
  // cluster tables: entries at or past the cluster count stay "not contracted"
  HEF_CHECK_CUDA(cudaMemsetAsync(ws.formed_by, 0xff, (size_t)(n + 1) * sizeof(int32_t), st));
  HEF_CHECK_CUDA(cudaMemsetAsync(ws.cflag, 0, (size_t)(n + 1) * sizeof(int), st));
  // Eq. R_W_update and Algorithm 1 step 6
  if (m > 0) {
    HEF_LAUNCH("k_update_r", st, k_update_r<<<grid_of(m), kThreads, 0, st>>>(
                                     mm, eptr, pins, R, eta, out->R_upd, ws.keys, ws.vals));
    HEF_CHECK_LAUNCH();
    HEF_PASS(sort_by_value(mm, out->R_upd, out->order, ws, st));
    HEF_LAUNCH("k_rank", st, k_rank<<<grid_of(m), kThreads, 0, st>>>(mm, out->order, eptr, ws.rank,
                                                                     ws.flag));
    HEF_CHECK_LAUNCH();
    HEF_PASS(exclusive_scan(ws.flag, ws.scan, m, ws.bsum, ws.counter, st));
  } else {
    HEF_CHECK_CUDA(cudaMemsetAsync(ws.scan, 0, sizeof(int), st));
  }
  HEF_LAUNCH("k_delta", st, k_delta<<<grid_of(m > 0 ? m : 1), kThreads, 0, st>>>(
                                mm, delta >= 0.0 ? delta : -1.0, quantile, out->order, out->R_upd,
                                ws.flag, ws.scan, out->delta));
  HEF_CHECK_LAUNCH();
  // Algorithm 2 step 5: greedy contraction
  HEF_LAUNCH("k_contract_init", st, k_contract_init<<<grid_of(N > 0 ? N : 1), kThreads, 0, st>>>(
                                        nn, mm, eptr, out->R_upd, out->delta, ws.state, ws.best,
                                        out->owner));
  HEF_CHECK_LAUNCH();
  if (m > 0) {
    int occ = 0;
    HEF_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_contract, kThreads, 0));
    const int grid = std::max(1, std::min(num_sms() * std::max(occ, 1), grid_of(m)));
    cudaError_t e = cudaSuccess;
    HEF_LAUNCH("k_contract", st,
               e = launch_cooperative_smem(k_contract, grid, kThreads, 0, st, mm, eptr, pins,
                                           (const int32_t*)ws.rank, ws.state, ws.best, out->owner,
                                           ws.last, ws.round_live, ws.counter + 1, ws.status));
    if (e != cudaSuccess) return set_error(HEF_ERR_CUDA, "k_contract: %s", cudaGetErrorString(e));
    HEF_LAUNCH("k_minpin", st, k_minpin<<<grid_of(m), kThreads, 0, st>>>(mm, eptr, pins, ws.state,
                                                                         ws.minpin));
    HEF_CHECK_LAUNCH();
  }
  // supernodes (numbered by their smallest vertex) and their weights
  int* cid = ws.scan;
  if (n > 0) {
    HEF_LAUNCH("k_cluster_flags", st, k_cluster_flags<<<grid_of(n), kThreads, 0, st>>>(
                                          nn, out->owner, ws.minpin, ws.flag));
    HEF_CHECK_LAUNCH();
  }
  HEF_PASS(exclusive_scan(ws.flag, cid, n, ws.bsum, ws.counter, st));
  if (n > 0) {
    HEF_LAUNCH("k_clusters", st, k_clusters<<<grid_of(n), kThreads, 0, st>>>(
                                     nn, out->owner, ws.minpin, cid, out->R_upd, eta, out->cluster,
                                     ws.eta_next, ws.formed_by, ws.cflag));
    HEF_CHECK_LAUNCH();
  }
  // nc is cid[n]; the clusters' arrays are indexed below it.  Algorithm 2
  // steps 7-10: local clustering of the isolated vertices
  HEF_CHECK_CUDA(cudaMemcpyAsync(ws.eta2, ws.eta_next, (size_t)(n > 0 ? n : 1) * sizeof(double),
                                 cudaMemcpyDeviceToDevice, st));
  if (n > 0) HEF_CHECK_CUDA(cudaMemsetAsync(out->target, 0xff, (size_t)n * sizeof(int32_t), st));
  if (n > 0) HEF_CHECK_CUDA(cudaMemsetAsync(out->dist, 0, (size_t)n * sizeof(double), st));
  int* nc_dev = cid + n;
  if (Q && n > 0 && m > 0) {
    // row of each contracted supernode in the centroid table (cflag is
    // defined for cluster ids below nc; the rest are never read)
    HEF_PASS(exclusive_scan(ws.cflag, ws.cflag, n, ws.bsum, ws.counter, st));
    const IncView g = view(inc);
    const int wgrid = (int)((n * 32 + kThreads - 1) / kThreads);
    auto run = [&](auto tag) -> hef_status {
      using QT = decltype(tag);
      // columns per lane: enough registers for K, no more than it needs
      auto cluster_seeds = [&](auto centroids, auto seeds) {
        HEF_LAUNCH("k_centroids", st, centroids<<<wgrid, kThreads, 0, st>>>(
                                          nn, ws.formed_by, ws.cflag, out->cluster, eptr, pins,
                                          static_cast<const QT*>(Q), ldq, K, QH, ws.mu, ws.mu32,
                                          ws.scale, ws.vinfo));
        HEF_LAUNCH("k_seeds", st, seeds<<<(int)((n * 32 + kSeedThreads - 1) / kSeedThreads), kSeedThreads, 0, st>>>(
                                      nn, out->owner, g.vptr, g.vedge, g.perm, eptr, pins, ws.vinfo,
                                      ws.mu, ws.mu32, ws.scale, static_cast<const QT*>(Q), ldq, K,
                                      QH, out->target, out->dist));
      };
      if (K <= 64) cluster_seeds(k_centroids<QT, 2>, k_seeds<QT, 2>);
      else if (K <= 128) cluster_seeds(k_centroids<QT, 4>, k_seeds<QT, 4>);
      else if (K <= 192) cluster_seeds(k_centroids<QT, 6>, k_seeds<QT, 6>);
      else if (K <= 256) cluster_seeds(k_centroids<QT, 8>, k_seeds<QT, 8>);
      else cluster_seeds(k_centroids<QT, 16>, k_seeds<QT, 16>);
      return HEF_OK;
    };
    if (dtype == HEF_F64) HEF_PASS(run(double{}));
    else if (dtype == HEF_BF16) HEF_PASS(run(__nv_bfloat16{}));
    else HEF_PASS(run(float{}));
    HEF_CHECK_LAUNCH();
    HEF_LAUNCH("k_merge_keys", st, k_merge_keys<<<grid_of(n), kThreads, 0, st>>>(
                                       nn, out->target, ws.keys, ws.vals));
    HEF_CHECK_LAUNCH();
    HEF_PASS(radix_sort(ws.keys, ws.vals, n, bits_for(n + 1), ws.sb, st));
    HEF_LAUNCH("k_merge_sums", st, k_merge_sums<<<grid_of(n), kThreads, 0, st>>>(
                                       nn, ws.keys, ws.vals, eta, out->dist, ws.eta2));
    HEF_CHECK_LAUNCH();
  }
  // final compact ids, their weights
  if (n > 0) {
    HEF_CHECK_CUDA(cudaMemsetAsync(ws.minv, 0x7f, (size_t)n * sizeof(int), st));
    HEF_LAUNCH("k_final_min", st, k_final_min<<<grid_of(n), kThreads, 0, st>>>(
                                      nn, out->cluster, out->target, ws.minv));
    HEF_LAUNCH("k_final_flags", st, k_final_flags<<<grid_of(n), kThreads, 0, st>>>(
                                        nn, out->cluster, out->target, ws.minv, ws.flag));
    HEF_CHECK_LAUNCH();
  }
  int* fid = ws.cflag;  // reuse: the centroid rows are no longer needed
  HEF_PASS(exclusive_scan(ws.flag, fid, n, ws.bsum, ws.counter, st));
  if (n > 0) {
    HEF_LAUNCH("k_final_ids", st, k_final_ids<<<grid_of(n), kThreads, 0, st>>>(
                                      nn, out->cluster, out->target, ws.minv, fid, ws.eta2,
                                      out->final_cluster, out->eta_out));
    HEF_CHECK_LAUNCH();
  }
  // Algorithm 2 step 6: the coarse hypergraph
  if (m > 0) {
    HEF_LAUNCH("k_coarse_count", st, k_coarse_count<<<grid_of(m), kThreads, 0, st>>>(
                                         mm, eptr, pins, out->final_cluster, ws.keep, ws.flag));
    HEF_CHECK_LAUNCH();
  }
  HEF_PASS(exclusive_scan(ws.keep, ws.ne, m, ws.bsum, ws.counter, st));
  HEF_PASS(exclusive_scan(ws.flag, ws.po, m, ws.bsum, ws.counter, st));
  HEF_LAUNCH("k_coarse_fill", st, k_coarse_fill<<<grid_of(m + 1), kThreads, 0, st>>>(
                                      mm, eptr, pins, w, out->final_cluster, ws.keep, ws.ne, ws.po,
                                      out->ceptr, out->cpins, out->cw, out->emap));
  HEF_LAUNCH("k_counts", st, k_counts<<<1, 32, 0, st>>>(nc_dev, fid + n, ws.ne + m, ws.po + m,
                                                         ws.status, out->counts));
  HEF_CHECK_LAUNCH();
  return HEF_OK;
}
