// knn_core.cuh -- choice of eps1 by the k-nearest-neighbours vote of
// Sec. 11, run by one warp, with no scratch memory.
//
// Each feature component is min-max scaled with the sample's min and max
// (Sec. 11.1; the query is not clamped; a constant component maps to 0).
// The squared Euclidean distance (Sec. 11.5) is summed over the selected
// components in index order.  The k nearest are the k smallest pairs
// (d2, index): one pass over the sample, 32 points at a time, keeps them as a
// sorted list spread over the warp's lanes, so that a distance, with its four
// FP64 divisions, is computed once.  Vote: weight 1/sqrt(d2) (Eq. 23) or 1 (Eq. 22), summed in
// selection order; when a selected neighbour is at distance 0 only the
// zero-distance neighbours vote, by count; ties go to the smallest class t.
// Every operation is an explicit IEEE-rounded intrinsic, so the result does
// not depend on compiler contraction.
#pragma once
#include <math.h>

#include "common.cuh"

namespace mpcg {

struct KnnSpec {
  const double* feat;  // [count][4], device
  const int8_t* cls;   // [count], device
  int count, k, weighted;
  unsigned mask;
  double fmin[4], fmax[4];
};

__device__ __forceinline__ double knn_scale(double v, double lo, double hi) {
  return hi > lo ? __ddiv_rn(__dsub_rn(v, lo), __dsub_rn(hi, lo)) : 0.0;
}

__device__ __forceinline__ double knn_d2(const KnnSpec& s, const double q[4], int i) {
  double d2 = 0.0;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (!((s.mask >> c) & 1u)) continue;
    const double p = knn_scale(s.feat[4 * (size_t)i + c], s.fmin[c], s.fmax[c]);
    const double diff = __dsub_rn(q[c], p);
    d2 = __dadd_rn(d2, __dmul_rn(diff, diff));
  }
  return d2;
}

// A sorted list of at most 64 pairs (d2, index), pair j in lane j & 31 (lo: j <
// 32, hi: the others).  Distances are kept as bit patterns: they are never
// negative, so their order as integers is that of the values, and an integer
// comparison does not wait for the FP64 pipe.  Unused places hold
// (infinity, 0x7fffffff), which no point equals.
struct KnnList {
  unsigned long long d_lo, d_hi;
  int i_lo, i_hi;
};
__device__ __forceinline__ void knn_clear(KnnList& L) {
  L.d_lo = L.d_hi = 0x7ff0000000000000ull;
  L.i_lo = L.i_hi = 0x7fffffff;
}
__device__ __forceinline__ bool knn_pair_less(unsigned long long d, int i, unsigned long long e, int j) {
  return d < e || (d == e && i < j);
}

// Insert one pair (the same in every lane); k > 32 uses the hi half.
__device__ __forceinline__ void knn_insert(KnnList& L, unsigned long long d, int i, int k) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned long long last_d = __shfl_sync(full, L.d_lo, 31);
  const int last_i = __shfl_sync(full, L.i_lo, 31);
  {
    const int at = __popc(__ballot_sync(full, knn_pair_less(L.d_lo, L.i_lo, d, i)));
    const unsigned long long ud = __shfl_up_sync(full, L.d_lo, 1);
    const int ui = __shfl_up_sync(full, L.i_lo, 1);
    if (lane > at) {
      L.d_lo = ud;
      L.i_lo = ui;
    } else if (lane == at) {
      L.d_lo = d;
      L.i_lo = i;
    }
    if (k <= 32) return;
    if (at < 32) {  // the pair pushed out of the lower half goes on
      d = last_d;
      i = last_i;
    }
  }
  const int at = __popc(__ballot_sync(full, knn_pair_less(L.d_hi, L.i_hi, d, i)));
  const unsigned long long ud = __shfl_up_sync(full, L.d_hi, 1);
  const int ui = __shfl_up_sync(full, L.i_hi, 1);
  if (lane > at) {
    L.d_hi = ud;
    L.i_hi = ui;
  } else if (lane == at) {
    L.d_hi = d;
    L.i_hi = i;
  }
}

// The k-th pair of the list (1 <= k <= 64), in every lane.
__device__ __forceinline__ void knn_kth(const KnnList& L, int k, unsigned long long& d, int& i) {
  const unsigned full = 0xffffffffu;
  const int j = (k - 1) & 31;
  const unsigned long long a = __shfl_sync(full, L.d_lo, j), b = __shfl_sync(full, L.d_hi, j);
  const int m = __shfl_sync(full, L.i_lo, j), n = __shfl_sync(full, L.i_hi, j);
  d = k <= 32 ? a : b;
  i = k <= 32 ? m : n;
}

// Enter one point per lane (`take`: the lane has one, d2 its distance) into
// the list; (td, ti) is the list's k-th pair.  NaN distances are never entered.
__device__ __forceinline__ void knn_enter(KnnList& L, bool take, double d2, int i, int k,
                                          unsigned long long& td, int& ti) {
  const unsigned full = 0xffffffffu;
  const unsigned long long bits = (unsigned long long)__double_as_longlong(d2);
  unsigned m = __ballot_sync(full, take && bits <= 0x7ff0000000000000ull && knn_pair_less(bits, i, td, ti));
  while (m) {  // warp-uniform
    const int src = __ffs(m) - 1;
    m &= m - 1;
    const unsigned long long d = __shfl_sync(full, bits, src);
    const int c = __shfl_sync(full, i, src);
    if (!knn_pair_less(d, c, td, ti)) continue;  // the threshold has moved
    knn_insert(L, d, c, k);
    knn_kth(L, k, td, ti);
  }
}

// The scaled query; false if a selected component is not finite.
__device__ __forceinline__ bool knn_query(const KnnSpec& s, const double chi[4], double q[4]) {
  bool good = s.count > 0 && s.k > 0 && s.k <= MPCG_KNN_MAX_K;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (((s.mask >> c) & 1u) && !isfinite(chi[c])) good = false;
    q[c] = knn_scale(chi[c], s.fmin[c], s.fmax[c]);
  }
  return good;
}

// The vote over the first k pairs of the list (k >= 1): the class, or -1 if a
// selected label is not a class.  Lane c keeps the score of class c.
__device__ __forceinline__ int knn_vote(const KnnSpec& s, const KnnList& L, int k) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int n_hi = k - 32;
  const int c_lo = lane < k ? s.cls[L.i_lo] : 0, c_hi = lane < n_hi ? s.cls[L.i_hi] : 0;
  if (__any_sync(full, c_lo < 0 || c_lo > 15 || c_hi < 0 || c_hi > 15)) return -1;
  const bool zero = __shfl_sync(full, L.d_lo, 0) == 0ull;  // only the neighbours at distance 0 vote
  auto weight = [&](unsigned long long d) -> double {
    if (zero) return d == 0ull ? 1.0 : 0.0;
    return s.weighted ? __ddiv_rn(1.0, __dsqrt_rn(__longlong_as_double((long long)d))) : 1.0;
  };
  const double w_lo = weight(L.d_lo);
  const double w_hi = n_hi > 0 ? weight(L.d_hi) : 0.0;
  double sc = 0.0;
  int present = 0;
  for (int j = 0; j < k; ++j) {  // in selection order
    const double w = __shfl_sync(full, j < 32 ? w_lo : w_hi, j & 31);
    const int c = __shfl_sync(full, j < 32 ? c_lo : c_hi, j & 31);
    const unsigned long long d = __shfl_sync(full, j < 32 ? L.d_lo : L.d_hi, j & 31);
    if (lane == c && (!zero || d == 0ull)) {
      sc = __dadd_rn(sc, w);
      present = 1;
    }
  }
  // the largest score, ties to the smallest class (scores are not negative)
  unsigned long long best = present ? (unsigned long long)__double_as_longlong(sc) : 0ull;
  int t = present ? lane : 99;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long e = __shfl_xor_sync(full, best, o);
    const int u = __shfl_xor_sync(full, t, o);
    if (u < 99 && (t == 99 || e > best || (e == best && u < t))) {
      best = e;
      t = u;
    }
  }
  return t < 99 ? t : -1;
}

// Class t in [0, 15] chosen for the raw query chi; -1 if the query, the
// sample or a label is invalid.  All 32 lanes of the warp must call it; the
// result is returned in every lane.
__device__ inline int knn_warp(const KnnSpec& s, const double chi[4]) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double q[4];
  if (!knn_query(s, chi, q)) return -1;
  const int k = s.k < s.count ? s.k : s.count;
  KnnList L;
  knn_clear(L);
  unsigned long long td = 0x7ff0000000000000ull;
  int ti = 0x7fffffff, bad = 0;
  for (int base = 0; base < s.count; base += 32) {
    const int i = base + lane;
    const double d2 = i < s.count ? knn_d2(s, q, i) : 0.0;
    if (d2 != d2) bad = 1;
    knn_enter(L, i < s.count, d2, i, k, td, ti);
  }
  if (__any_sync(full, bad)) return -1;
  return knn_vote(s, L, k);
}

// eps1 = 10^-t as the correctly rounded decimal literal.
__device__ __forceinline__ double pow10_neg(int t) {
  switch (t) {
    case 0: return 1e0;
    case 1: return 1e-1;
    case 2: return 1e-2;
    case 3: return 1e-3;
    case 4: return 1e-4;
    case 5: return 1e-5;
    case 6: return 1e-6;
    case 7: return 1e-7;
    case 8: return 1e-8;
    case 9: return 1e-9;
    case 10: return 1e-10;
    case 11: return 1e-11;
    case 12: return 1e-12;
    case 13: return 1e-13;
    case 14: return 1e-14;
    default: return 1e-15;
  }
}

}  // namespace mpcg
